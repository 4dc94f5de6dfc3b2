// Lattice graphs on the host side: detection, placement of the tiled state, launch
// (the kernels: mf_lattice2.cu, mf_lattice3.cu).
#include <limits.h>
#include <string.h>

#include "mf_internal.h"
#include "mf_lattice.cuh"

namespace mf {

const void *lattice2_fn();
const void *lattice3_fn();
size_t lattice3_smem();
size_t lattice_queue_bytes(int tiles);

namespace {

// ------------------------------------------------------------------ detection

// out[0]: smallest |difference| above 1 between the cell indices of an arc's
// ends (INT_MAX: none), out[1]: the largest.
__global__ void k_lat_strides(int n, const int *row, const int *head, Lat L, int *out) {
  int lo = INT_MAX, hi = 0;
  for (int v = blockIdx.x * blockDim.x + threadIdx.x; v < n; v += gridDim.x * blockDim.x) {
    if (v == L.s || v == L.t) continue;
    const int p = cell_of(L, v), e = row[v + 1];
    for (int a = row[v]; a < e; a++) {
      const int w = head[a];
      if (w == L.s || w == L.t) continue;
      const int x = abs(cell_of(L, w) - p);
      hi = max(hi, x);
      if (x > 1) lo = min(lo, x);
    }
  }
  lo = __reduce_min_sync(LFULL, lo);
  hi = __reduce_max_sync(LFULL, hi);
  if ((threadIdx.x & 31) == 0) {
    if (lo < INT_MAX) atomicMin(&out[0], lo);
    if (hi > 0) atomicMax(&out[1], hi);
  }
}

// Sets *bad when some arc does not join neighbouring cells of the X x Y x Z box
// (or a cell and a terminal), a cell has two slots in one direction or to one
// terminal, or s and t are joined directly, to each other or to themselves (the
// outputs of terminals are written from the cells' slots).
__global__ void k_lat_check(int n, const int *row, const int *head, Lat L, int *bad) {
  bool f = false;
  const int A = L.X, B = L.X * L.Y;
  for (int v = blockIdx.x * blockDim.x + threadIdx.x; v < n; v += gridDim.x * blockDim.x) {
    if (v == L.s || v == L.t) continue;
    const int p = cell_of(L, v), e = row[v + 1];
    unsigned seen = 0;
    for (int a = row[v]; a < e; a++) {
      const int w = head[a];
      unsigned bit;
      if (w == L.s || w == L.t) {
        bit = w == L.s ? 1u : 2u;
      } else {
        const int q = cell_of(L, w), x = q - p, y = abs(x);
        if (y == 1 && p / A == q / A)
          bit = 4u << (x > 0);
        else if (y == A && (L.dim == 2 || p / B == q / B))
          bit = 16u << (x > 0);
        else if (L.dim == 3 && y == B)
          bit = 64u << (x > 0);
        else {
          f = true;
          break;
        }
      }
      if (seen & bit) f = true;
      seen |= bit;
    }
  }
  const int tid = blockIdx.x * blockDim.x + threadIdx.x;
  for (int k = 0; k < 2; k++) {
    const int v = k ? L.t : L.s;
    for (long long a = (long long)row[v] + tid; a < row[v + 1]; a += gridDim.x * blockDim.x)
      if (head[a] == L.t || head[a] == L.s) f = true;
  }
  if (__any_sync(LFULL, f) && (threadIdx.x & 31) == 0) atomicOr(bad, 1);
}

}  // namespace

// Options a lattice solve takes: the improved rounds with CTA-local lists, the
// time-based relabel trigger (its only one) and the default CTA. Anything that
// names a part of the list solver (simple rounds, gap relabeling, a round limit,
// another CTA size, register budget or degree bin) runs there.
bool lattice_applies(const mf_graph *g, const mf_options &o) {
  return g->lat.dim && !o.simple_rounds && !o.gap_every && o.max_rounds == 0 && o.gr_time_ratio > 0 && o.block_threads == LT &&
         o.kernel_variant == 0 && keep_local_limit(o, g->max_degree, o.block_threads) > 0;
}

// Places the tiled state in the list solver's arrays (both set their state up
// from the capacities on every solve), or in a buffer of its own where the
// padding of the last tiles makes it larger than those.
static int lattice_place(mf_graph *g) {
  Lat &L = g->lat;
  const size_t cells = (size_t)L.tiles * TV, nd = 2 * (size_t)L.dim;
  const size_t faces = (size_t)L.tiles * nd * (L.dim == 3 ? 64 : 32);
  char *res = reinterpret_cast<char *>(g->rr), *vert = reinterpret_cast<char *>(g->vs);
  char *bfs = reinterpret_cast<char *>(g->blab);
  int *list[3] = {g->list[0], g->list[1], g->list[2]};
  const size_t nres = cells * nd * 4, nvert = cells * (L.dim == 3 ? 21 : 20), nbfs = faces * 4 + cells * 2;
  const size_t queue = lattice_queue_bytes(L.tiles);
  if (nres > (size_t)g->m * 8 || nvert > (size_t)g->n * sizeof(VRec) || nbfs > (size_t)g->n * 8 ||
      2 * queue > (size_t)g->n * 4) {
    const int rc = galloc(g, &g->lat_buf, nres + nvert + nbfs + 2 * queue + (size_t)L.tiles * 12, "cudaMalloc lattice state");
    if (rc) return rc;
    res = reinterpret_cast<char *>(g->lat_buf);
    vert = res + nres;
    bfs = vert + nvert;
    list[0] = reinterpret_cast<int *>(bfs + nbfs);
    list[1] = list[0] + queue / 4;
    list[2] = list[1] + queue / 4;
  }
  L.r = reinterpret_cast<int *>(res);
  L.ex = reinterpret_cast<long long *>(vert);
  L.d = reinterpret_cast<int *>(L.ex + cells);
  L.drain = L.d + cells;
  L.back = L.drain + cells;
  L.slots = reinterpret_cast<unsigned char *>(L.back + cells);
  L.inbox = reinterpret_cast<int *>(bfs);
  L.mask = reinterpret_cast<unsigned char *>(L.inbox + faces);
  L.ret = L.mask + cells;
  L.list[0] = list[0];
  L.list[1] = list[1];
  L.state = list[2];
  L.bits = L.state + L.tiles;
  return MF_OK;
}

// Gives the buffer of the tiled state back.
static void lattice_unplace(mf_graph *g) {
  gfree(g, g->lat_buf);
  g->lat_buf = nullptr;
  g->lat.r = nullptr;
}

// Called whenever g's options are set: the tiled state has its place while they
// ask for lattice solves (a buffer of its own only then). Without memory for it
// the list solver takes the graph from then on.
void lattice_options(mf_graph *g) {
  if (!g->lat.dim) return;
  if (!lattice_applies(g, g->opt)) {
    if (g->lat_buf) lattice_unplace(g);
  } else if (!g->lat.r && lattice_place(g) != MF_OK) {
    clear_error();
    g->lat.dim = 0;
  }
}

// Where memory for a solve's outputs is short: gives the buffer of the tiled state
// back and leaves g to the list solver. False if there is none.
bool lattice_give_up(mf_graph *g) {
  if (!g->lat_buf) return false;
  lattice_unplace(g);
  g->lat.dim = 0;
  return true;
}

// Decides whether g (validated, on the device) is a lattice and sets the geometry in
// g->lat (dim 0: it is not). Unions, of one instance too, run the list solver and are not
// looked at. `scratch`: two ints of device memory.
int lattice_detect(mf_graph *g, int *scratch, cudaStream_t st) {
  memset(&g->lat, 0, sizeof(g->lat));
  if (g->vinst || g->max_degree > 8 || g->m == 0) return MF_OK;
  Lat L;
  memset(&L, 0, sizeof(L));
  L.s = g->s;
  L.t = g->t;
  L.cells = g->n - 2;
  const int T = 256;
  const int G = (int)(((long long)g->n + T - 1) / T < 4096 ? ((long long)g->n + T - 1) / T : 4096);
  int h[2] = {INT_MAX, 0};
  cudaError_t e = cudaMemcpyAsync(scratch, h, 8, cudaMemcpyHostToDevice, st);
  if (e == cudaSuccess) {
    k_lat_strides<<<G, T, 0, st>>>(g->n, g->row, g->head, L, scratch);
    e = cudaMemcpyAsync(h, scratch, 8, cudaMemcpyDeviceToHost, st);
  }
  if (e == cudaSuccess) e = cudaStreamSynchronize(st);
  if (e != cudaSuccess) return cuda_fail(e, "lattice check");
  if (h[0] == INT_MAX || h[0] < 2 || h[1] % h[0]) return MF_OK;
  L.dim = h[1] == h[0] ? 2 : 3;
  L.X = h[0];
  L.Y = L.dim == 2 ? (L.cells + L.X - 1) / L.X : h[1] / h[0];
  L.Z = L.dim == 2 ? 1 : (int)(((long long)L.cells + h[1] - 1) / h[1]);
  if (L.dim == 3 && L.Y < 2) return MF_OK;
  L.TX = (L.X + (L.dim == 3 ? 7 : 31)) / (L.dim == 3 ? 8 : 32);
  L.TY = (L.Y + (L.dim == 3 ? 7 : 15)) / (L.dim == 3 ? 8 : 16);
  L.TZ = L.dim == 3 ? (L.Z + 7) / 8 : 1;
  const long long tiles = (long long)L.TX * L.TY * L.TZ;
  if (tiles > INT_MAX / TV) return MF_OK;
  L.tiles = (int)tiles;
  // Thin boxes are mostly padding, and tiles cost time and memory by their padded size. Measured, lattice against
  // list solver on boxes of 600 to 1,000,000 cells and 2 to 40 cells a side: up to 4 padded cells per cell (3.5 in
  // 3D) the lattice solver is 1.3 to 3 times as fast at every size; beyond, 1.1 to 2 times up to some 1,500 tiles,
  // but 0.7 to 1.1 times at 10,000 to 30,000 tiles.
  const long long padded = tiles * TV;
  if (2 * padded > (L.dim == 2 ? 8LL : 7LL) * L.cells + 16 * TV && (tiles > 2048 || padded > 8LL * L.cells + 8 * TV)) return MF_OK;
  e = cudaMemsetAsync(scratch, 0, 4, st);
  if (e == cudaSuccess) {
    k_lat_check<<<G, T, 0, st>>>(g->n, g->row, g->head, L, scratch);
    e = cudaMemcpyAsync(h, scratch, 4, cudaMemcpyDeviceToHost, st);
  }
  if (e == cudaSuccess) e = cudaStreamSynchronize(st);
  if (e != cudaSuccess) return cuda_fail(e, "lattice check");
  if (!h[0]) g->lat = L;
  return MF_OK;
}

// CTAs of a lattice solve. Images: as many as fit, at most one per tile.
// Volumes: one per SM, at most one per 4 tiles (one warp per scheduler); CTAs
// without a tile would only lengthen the grid barriers.
int lattice_grid(const mf_graph *g, int sms, int *grid) {
  const bool flat = g->lat.dim == 2;
  const void *fn = flat ? lattice2_fn() : lattice3_fn();
  const size_t smem = flat ? 0 : lattice3_smem();
  cudaError_t e = cudaSuccess;
  if (smem) e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  int bps = 0;
  if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&bps, fn, LT, smem);
  if (e != cudaSuccess) return cuda_fail(e, "lattice solver occupancy");
  if (bps < 1) return fail(MF_ERR_CUDA, "lattice solver does not fit an SM");
  if (g->opt.blocks_per_sm > 0 && g->opt.blocks_per_sm < bps) bps = g->opt.blocks_per_sm;
  const long long most = (long long)bps * sms, want = flat ? g->lat.tiles : ((long long)g->lat.tiles + 3) / 4;
  *grid = (int)(want < most ? want : most);
  return MF_OK;
}

cudaError_t launch_lattice(const Dev &D, int grid, cudaStream_t stream) {
  Dev d = D;
  void *args[] = {&d};
  const bool flat = D.lat.dim == 2;
  return cudaLaunchCooperativeKernel(flat ? lattice2_fn() : lattice3_fn(), dim3(grid), dim3(LT), args,
                                     flat ? 0 : lattice3_smem(), stream);
}

}  // namespace mf
