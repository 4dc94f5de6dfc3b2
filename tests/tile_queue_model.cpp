// The tile queue of the volume solver (csrc/mf_tile_queue.cuh) under a model of the GPU's memory order: warps are
// coroutines that a seeded scheduler switches at every memory operation, some of them held up for long, and vector
// clocks follow what fences and atomics order. Prints "ok", or what went wrong:
//   race    a visit of a tile does not come after the last one, or not after the amounts it was woken for
//   twice   two warps visit one tile at a time
//   lost    work that nobody visits (the warps wait for ever)
// argv: tiles warps visits seed mode hold (turns a warp is held up for, at most). Mode 0: the queue as it is; 1: entries are made without a release; 2: entries
// overwrite what lies in their place; 3: any ticket of a place takes its entry.
#include <stddef.h>
#include <stdio.h>
#include <stdlib.h>
#include <ucontext.h>

#include <map>
#include <random>
#include <vector>

#include "mf_tile_queue.cuh"

namespace {

using Clock = std::vector<unsigned>;
int nwarps, mode, hold, cur = -1;
std::mt19937 rng;
ucontext_t main_ctx;
std::vector<ucontext_t> ctx;
std::vector<int> asleep;  // turns a warp is held up for
std::vector<bool> over;
std::vector<Clock> now, seen, out;  // per warp: clock; joined by its next acquire fence; released by its last fence
std::map<const void *, Clock> at;   // per location: what an acquire that reads it is ordered after

[[noreturn]] void fail(const char *what) {
  printf("%s\n", what);
  fflush(stdout);
  exit(0);
}
void join(Clock &a, const Clock &b) {
  for (size_t i = 0; i < b.size(); i++)
    if (b[i] > a[i]) a[i] = b[i];
}
Clock &loc(const void *p) {
  Clock &c = at[p];
  c.resize((size_t)nwarps);
  return c;
}
void turn() {  // back to the scheduler
  now[cur][cur]++;
  swapcontext(&ctx[cur], &main_ctx);
}
void fence() {
  join(now[cur], seen[cur]);
  out[cur] = now[cur];
}

// An amount a warp put into an inbox; told[id]: the tile's state word says so.
struct Amount {
  int by;
  unsigned clk;
  size_t id;
};
std::vector<char> told;
std::vector<size_t> telling;  // told by the next RMW

struct Mem {
  template <class T, class F>
  T rmw(T *p, bool acquire, F f) {
    const std::vector<size_t> say = std::move(telling);
    telling.clear();
    turn();
    for (size_t id : say) told[id] = 1;
    const T old = *p;
    Clock &c = loc(p);
    join(seen[cur], c);
    if (acquire) join(now[cur], c);
    join(c, out[cur]);  // an RMW continues the release sequence it reads from
    *p = f(old);
    return old;
  }
  int add(int *p, int x) { return rmw(p, false, [x](int o) { return o + x; }); }
  int or_relaxed(int *p, int x) { return rmw(p, false, [x](int o) { return o | x; }); }
  int or_acquire(int *p, int x) { return rmw(p, true, [x](int o) { return o | x; }); }
  int and_acquire(int *p, int x) { return rmw(p, true, [x](int o) { return o & x; }); }
  int exch_acquire(int *p, int x) { return rmw(p, true, [x](int) { return x; }); }
  unsigned cas(unsigned *p, unsigned expect, unsigned x) {
    if (mode == 2) {
      store(p, x);
      return 0;
    }
    return rmw(p, false, [expect, x](unsigned o) { return o == expect ? x : o; });
  }
  unsigned load(unsigned *p) {
    turn();
    join(seen[cur], loc(p));
    return *p;
  }
  void store(unsigned *p, unsigned x) {
    turn();
    loc(p) = out[cur];
    *p = x;
  }
  void release() {
    if (mode != 1) fence();
  }
  void acquire() { fence(); }
  bool wait(unsigned spins) {
    if (spins > 1000000) fail("lost");
    return true;
  }
};

int tiles, visits_left;
std::vector<unsigned> ring;
std::vector<int> state, visiting, writer;
std::vector<unsigned> wrote;                               // clock of the writer's last write of the tile
std::vector<std::vector<Amount>> inbox;                    // per tile and face
int head, tail, idle;
bool done = false;

mf::TileQueue<Mem> queue() { return {ring.data(), &head, &tail, state.data(), tiles, Mem{}}; }

// A tile's visit: its cells are read and written, and some neighbours get an amount.
void visit(int t) {
  mf::TileQueue<Mem> q = queue();
  // the tile's cells are read before the exchange returns
  if (writer[t] >= 0 && now[cur][writer[t]] < wrote[t]) fail("race");
  if (visiting[t]++) fail("twice");
  const int faces = q.begin(t) >> mf::FACES;
  for (int j = 0; j < 6; j++)
    if ((faces >> j) & 1) {
      std::vector<Amount> untold;
      for (const Amount &a : inbox[(size_t)t * 6 + j])
        if (!told[a.id])
          untold.push_back(a);
        else if (now[cur][a.by] < a.clk)
          fail("race");
      inbox[(size_t)t * 6 + j] = untold;
    }
  turn();
  if (rng() % 4 == 0) asleep[cur] = (int)(rng() % (unsigned)(hold / 400 + 1));
  turn();
  writer[t] = cur;
  wrote[t] = now[cur][cur];
  int wake[2], n = 0;  // offset of the tile across face k: k + 1
  bool again = false;
  if (visits_left > 0) {
    visits_left--;
    again = rng() % 16 != 0;
    for (; n < 2 && tiles > 1 && rng() % 3 == 0; n++) wake[n] = (int)(rng() % (tiles > 6 ? 6 : tiles - 1));
    for (int k = 0; k < n; k++) {  // (the amounts themselves are atomics)
      inbox[(size_t)((t + wake[k] + 1) % tiles) * 6 + wake[k]].push_back({cur, now[cur][cur], told.size()});
      told.push_back(0);
    }
  }
  visiting[t]--;
  turn();
  fence();
  for (int k = 0; k < n; k++) {
    const int x = (t + wake[k] + 1) % tiles;
    for (const Amount &a : inbox[(size_t)x * 6 + wake[k]])
      if (a.by == cur) telling.push_back(a.id);
    if (q.mark(x, 1 << wake[k])) q.push(x, true);
  }
  if (q.end(t, again)) q.push(t, false);
}

void warp() {
  mf::TileQueue<Mem> q = queue();
  for (;;) {
    const unsigned ticket = q.ticket();
    auto look = [&]() {
      if (mode != 3) return q.look(ticket);
      const unsigned v = q.m.load(q.place(ticket));
      return v ? (int)(v & ((1u << mf::Q_TILE_BITS) - 1)) - 1 : -1;
    };
    int t = look();
    if (t < 0) {
      idle++;
      for (unsigned spins = 0;; spins++) {
        if (rng() % 64 == 0) asleep[cur] = (int)(rng() % (unsigned)(hold + 1));  // a long sleep between two looks
        turn();
        t = look();
        if (t >= 0 || done) break;
        if (idle == nwarps && head == tail + nwarps) done = true;
        if (spins > 3000000) fail("lost");
      }
      if (t < 0) break;
      idle--;
    }
    if (rng() % 8 == 0) {
      asleep[cur] = (int)(rng() % (unsigned)(hold / 10 + 1));
      turn();
    }
    q.take(ticket);
    visit(t);
  }
  over[cur] = true;
  for (;;) swapcontext(&ctx[cur], &main_ctx);
}

}  // namespace

int main(int argc, char **argv) {
  if (argc < 7) return 2;
  tiles = atoi(argv[1]);
  nwarps = atoi(argv[2]);
  visits_left = atoi(argv[3]);
  rng.seed((unsigned)atoi(argv[4]));
  mode = atoi(argv[5]);
  hold = atoi(argv[6]);
  ring.assign((size_t)mf::q_slots(tiles) * mf::Q_STRIDE, 0);
  state.assign((size_t)tiles, 0);
  visiting.assign((size_t)tiles, 0);
  writer.assign((size_t)tiles, -1);
  wrote.assign((size_t)tiles, 0);
  inbox.assign((size_t)tiles * 6, {});
  now.assign((size_t)nwarps, Clock((size_t)nwarps, 0));
  seen = out = now;
  for (int t = 0; t < tiles; t++) {  // queued before the phase (a grid barrier orders this before everything)
    state[t] = mf::QUEUED;
    *queue().place((unsigned)t) = queue().entry((unsigned)t, t);
  }
  tail = tiles;
  std::vector<std::vector<char>> stack((size_t)nwarps, std::vector<char>(1 << 16));
  ctx.resize((size_t)nwarps);
  asleep.assign((size_t)nwarps, 0);
  over.assign((size_t)nwarps, false);
  for (int w = 0; w < nwarps; w++) {
    getcontext(&ctx[w]);
    ctx[w].uc_stack.ss_sp = stack[w].data();
    ctx[w].uc_stack.ss_size = stack[w].size();
    ctx[w].uc_link = &main_ctx;
    makecontext(&ctx[w], warp, 0);
  }
  for (long long steps = 0;; steps++) {
    if (steps > 20000000) fail("lost");
    std::vector<int> can;
    bool left = false;
    for (int w = 0; w < nwarps; w++) {
      if (over[w]) continue;
      left = true;
      if (asleep[w] > 0)
        asleep[w]--;
      else
        can.push_back(w);
    }
    if (!left) break;
    if (can.empty()) continue;
    cur = can[rng() % can.size()];
    swapcontext(&main_ctx, &ctx[cur]);
  }
  for (int t = 0; t < tiles; t++)
    if (state[t]) fail("lost");
  puts("ok");
  return 0;
}
