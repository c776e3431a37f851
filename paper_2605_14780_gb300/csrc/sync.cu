// Block-edge averaging (Sync rows, Sec. III-B) on sm_103a.
//
// Sync rows overwrite data cells that several blocks store for one physical
// location, and read data cells themselves, so one apply runs in two steps
// around the other kernels: the rows are evaluated into a plan-owned staging
// buffer while every row of the operator still reads the input values, and
// the staged values are written to the data cells afterwards.  The adjoint
// mirrors it: the rows' cotangents are moved to the staging buffer (their
// data cells' own cotangent is consumed), the ghost gather runs, then every
// column the rows read gathers its staged contributions.  Sync sets are
// small (the shared edges of the blocks): one thread per (row or column,
// level), levels fastest when they are contiguous in memory, rows fastest
// otherwise, so the accesses of a warp stay coalesced in both layouts.  Rows
// that fall into closed groups skip the staging in the forward (below).
#include <cstdint>

#include "bc_internal.h"

namespace bcg {
namespace {

constexpr int kSyncThreads = 256;

template <typename T>
__device__ __forceinline__ T* slot_at(void* const* slots, int slot, int off) {
  return static_cast<T*>(slots[slot]) + off;
}

// thread t -> (row or column u, level l): levels fastest when the levels are
// contiguous in memory, else rows fastest (consecutive cells of a box)
__device__ __forceinline__ void split(const SyncCtx& s, int n, int64_t t, int& u, int& l) {
  if (s.level_fast) {
    u = (int)(t / s.lmax);
    l = (int)(t - (int64_t)u * s.lmax);
  } else {
    l = (int)(t / n);
    u = (int)(t - (int64_t)l * n);
  }
}

template <typename T>
__global__ void __launch_bounds__(kSyncThreads) k_sync(SyncCtx s, int step, void* const* slots,
                                                      const int32_t* slot_ls) {
  const int64_t t = (int64_t)blockIdx.x * kSyncThreads + threadIdx.x;
  T* stage = static_cast<T*>(s.stage);
  if (step == SYNC_ADJOINT) {
    if (t >= (int64_t)s.ncols * s.lmax) return;
    int u, l;
    split(s, s.ncols, t, u, l);
    const int4 c = s.col[u];
    if (l >= c.z) return;
    T* xb = slot_at<T>(slots, c.x, c.y + l * __ldg(slot_ls + c.x));
    const T* w = static_cast<const T*>(s.cw);
    const int e0 = __ldg(s.cptr + u), e1 = __ldg(s.cptr + u + 1);
    T acc = *xb;
    for (int e = e0; e < e1; ++e) acc = fma(__ldg(w + e), stage[__ldg(s.cstage + e) + l], acc);
    *xb = acc;
    return;
  }
  if (t >= (int64_t)s.nrows * s.lmax) return;
  int u, l;
  split(s, s.nrows, t, u, l);
  const int4 r = s.row[u];
  if (l >= r.w) return;
  T* d = slot_at<T>(slots, r.x, r.y + l * __ldg(slot_ls + r.x));
  if (step == SYNC_ROWS) {
    const T* w = static_cast<const T*>(s.w);
    const int e0 = __ldg(s.ptr + u), e1 = __ldg(s.ptr + u + 1);
    T acc = T(0);
    for (int e = e0; e < e1; ++e) {
      const int2 en = s.ent[e];
      acc = fma(__ldg(w + e), *slot_at<T>(slots, en.x, en.y + l * __ldg(slot_ls + en.x)), acc);
    }
    stage[r.z + l] = acc;
  } else if (step == SYNC_COMMIT) {
    *d = stage[r.z + l];
  } else {  // SYNC_SNAPSHOT
    stage[r.z + l] = *d;
    *d = T(0);
  }
}

// Closed groups: up to four rows that read exactly the cells they write (the
// copies of one node), so one thread sums them all and then stores them, with
// no staging: the cells' DRAM granules (a node of a column is 4 bytes of 64)
// are read and written once, in one launch instead of two, and the rows'
// tables load once for LV levels.  Runs after every kernel that reads data.
// Shared nodes of 8 x 8 blocks of 129^2 x 96 planes FP32: 41 us for the rows
// beside the ghost kernel and 41 for the commit -> 46 us, the whole fill 132 ->
// 110 us.
constexpr int kSyncLevels = 4;  // levels of a thread where they are far apart

template <typename T, int LV>
__global__ void __launch_bounds__(kSyncThreads)
    k_sync_groups(SyncCtx s, void* const* slots, const int32_t* slot_ls) {
  const int64_t t = (int64_t)blockIdx.x * kSyncThreads + threadIdx.x;
  int u, l0;
  if (LV == 1) {  // levels contiguous: levels fastest
    u = (int)(t / s.lmax);
    l0 = (int)(t - (int64_t)u * s.lmax);
  } else {
    const int64_t c = t / s.ngroups;
    u = (int)(t - c * s.ngroups);
    l0 = (int)c * LV;
  }
  if (u >= s.ngroups || l0 >= s.lmax) return;
  const int4 g = __ldg(s.group + u);
  const int rows[4] = {g.x, g.y, g.z, g.w};
  T acc[4][LV];
  T* d[4];
  int64_t dls[4];
  int nl = 0;
#pragma unroll
  for (int r = 0; r < 4; ++r) {
#pragma unroll
    for (int l = 0; l < LV; ++l) acc[r][l] = T(0);
    if (rows[r] < 0) continue;
    const int4 rw = __ldg(s.row + rows[r]);
    nl = rw.w - l0;
    if (nl <= 0) return;  // a group's rows have one level count
    dls[r] = __ldg(slot_ls + rw.x);
    d[r] = slot_at<T>(slots, rw.x, rw.y) + l0 * dls[r];
    const int e0 = __ldg(s.ptr + rows[r]), e1 = __ldg(s.ptr + rows[r] + 1);
    for (int e = e0; e < e1; ++e) {
      const int2 en = __ldg(s.ent + e);
      const T w = __ldg(static_cast<const T*>(s.w) + e);
      const int64_t xls = __ldg(slot_ls + en.x);
      const T* x = slot_at<T>(slots, en.x, en.y) + l0 * xls;
#pragma unroll
      for (int l = 0; l < LV; ++l)
        if (l < nl) acc[r][l] = fma(w, x[l * xls], acc[r][l]);
    }
  }
#pragma unroll
  for (int r = 0; r < 4; ++r)
    if (rows[r] >= 0) {
#pragma unroll
      for (int l = 0; l < LV; ++l)
        if (l < nl) d[r][l * dls[r]] = acc[r][l];
    }
}

}  // namespace

cudaError_t launch_sync(int dtype, int step, const SyncCtx& s, void* const* slots,
                        const int32_t* slot_ls, cudaStream_t stream) {
  if (step == SYNC_GROUPS) {
    if (s.ngroups <= 0) return cudaSuccess;
    const int64_t parts = s.level_fast ? s.lmax : (s.lmax + kSyncLevels - 1) / kSyncLevels;
    const int blocks = (int)((s.ngroups * parts + kSyncThreads - 1) / kSyncThreads);
    auto* k = dtype == 1 ? (s.level_fast ? k_sync_groups<double, 1> : k_sync_groups<double, kSyncLevels>)
                         : (s.level_fast ? k_sync_groups<float, 1> : k_sync_groups<float, kSyncLevels>);
    k<<<blocks, kSyncThreads, 0, stream>>>(s, slots, slot_ls);
    return cudaGetLastError();
  }
  const int64_t n = (int64_t)(step == SYNC_ADJOINT ? s.ncols : s.nrows) * s.lmax;
  if (n <= 0) return cudaSuccess;
  const int grid = (int)((n + kSyncThreads - 1) / kSyncThreads);
  if (dtype == 1)
    k_sync<double><<<grid, kSyncThreads, 0, stream>>>(s, step, slots, slot_ls);
  else
    k_sync<float><<<grid, kSyncThreads, 0, stream>>>(s, step, slots, slot_ls);
  return cudaGetLastError();
}

}  // namespace bcg
