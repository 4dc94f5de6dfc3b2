#pragma once
// Index checks of the gathers (a build with MF_CHECK_BOUNDS, for tests): an
// index outside its array is recorded in the error word (MF_ERR_INTERNAL, the
// source file and line in err_where and the index in bad_index, first one wins)
// and replaced by 0, so the access stays inside the array and the solve ends
// at its next grid barrier; no trap. Without MF_CHECK_BOUNDS the macros are the
// index itself. A file that uses them sets MF_FILE, its place in check_files
// (mf_api.cu).
#include "mf.h"
#include "mf_device.cuh"

#ifdef MF_CHECK_BOUNDS
namespace mf {
static __device__ __noinline__ long long mf_bad_index(const Dev &D, long long i, int where) {
  if (atomicCAS(&D.ctl->err, 0, MF_ERR_INTERNAL) == 0) {
    atomicExch(&D.ctl->err_where, where);
    atomicExch(reinterpret_cast<unsigned long long *>(&D.ctl->bad_index), (unsigned long long)i);
  }
  return 0;
}
}  // namespace mf
#define MF_CHECKED(D, i, lim) \
  (((unsigned long long)(long long)(i) < (unsigned long long)(long long)(lim)) ? (i) \
      : (decltype((i) + 0))mf::mf_bad_index(D, (long long)(i), mf::CHECK_WHERE + mf::CHECK_LINES * MF_FILE + __LINE__))
#else
#define MF_CHECKED(D, i, lim) (i)
#endif

// slots, vertices and row offsets
#define MF_SLOT(D, a) MF_CHECKED(D, a, (D).m)
#define MF_VTX(D, v) MF_CHECKED(D, v, (D).n)
#define MF_ROW(D, v) MF_CHECKED(D, v, (D).n + 1)
// lattices: tiles, face bits by sweep parity, per-cell arrays, residuals by tile and direction, inbox entries, and
// labels of a tile with its halo in shared memory
#define MF_TILE(D, t) MF_CHECKED(D, t, (D).lat.tiles)
#define MF_BITS(D, i) MF_CHECKED(D, i, 2LL * (D).lat.tiles)
#define MF_CELL(D, i) MF_CHECKED(D, i, (long long)(D).lat.tiles * TV)
#define MF_RES(D, i) MF_CHECKED(D, i, (long long)(D).lat.tiles * TV * Geo<DIM>::ND)
#define MF_INBOX(D, i) MF_CHECKED(D, i, (long long)(D).lat.tiles * Geo<DIM>::NH)
#define MF_LAB(D, i) MF_CHECKED(D, i, Geo<DIM>::PAD)
