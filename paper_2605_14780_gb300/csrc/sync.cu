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
// copies of one node), so one thread sums them all at one level and then
// stores them, with no staging: the cells' DRAM granules (a node of a column is
// 4 bytes of 64) are read and written once, in one launch instead of two.  Runs
// after every kernel that reads data.  Bound by DRAM granules on large grids
// and by its chain of dependent loads on small ones, so a group comes as a
// record (SyncCtx::group): record, slot pointers, values is the whole chain,
// each distinct cell is loaded once, and the rows are summed from registers in
// entry order.  One level a thread and CTAs of 64 threads spread a small grid
// over the SMs (four levels a thread, which saves table loads: within 2 % on
// large grids, 30 % slower on small FP64 ones, whose multiply-adds then queue on
// a few SMs).
// 8 x 8 blocks of 129^2 x 96 planes FP32, the whole fill: 133 us staged, 99 with
// the rows' own tables walked in series, 90 so; 2 x 2 blocks of 9^2 x 2 planes
// FP64: 5.8, 9.3, 5.3 us.
constexpr int kGroupThreads = 64;

template <typename T>
__device__ __forceinline__ void load_row_weights(const T* p, T (&w)[kSyncGroup]) {
  if constexpr (sizeof(T) == 4) {
    const float4 v = __ldg(reinterpret_cast<const float4*>(p));
    w[0] = v.x;
    w[1] = v.y;
    w[2] = v.z;
    w[3] = v.w;
  } else {
    const double2 v = __ldg(reinterpret_cast<const double2*>(p));
    const double2 u = __ldg(reinterpret_cast<const double2*>(p) + 1);
    w[0] = v.x;
    w[1] = v.y;
    w[2] = u.x;
    w[3] = u.y;
  }
}

template <typename T>
__global__ void __launch_bounds__(kGroupThreads) k_sync_groups(SyncCtx s, void* const* slots) {
  const int64_t t = (int64_t)blockIdx.x * kGroupThreads + threadIdx.x;
  if (t >= (int64_t)s.ngroups * s.lmax) return;
  int u, l;
  split(s, s.ngroups, t, u, l);
  const int64_t ng = s.ngroups;
  const int4 sl = __ldg(s.group + u), of = __ldg(s.group + ng + u), st = __ldg(s.group + 2 * ng + u),
             me = __ldg(s.group + 3 * ng + u);
  const int slot[kSyncGroup] = {sl.x, sl.y, sl.z, sl.w}, off[kSyncGroup] = {of.x, of.y, of.z, of.w};
  const int ls[kSyncGroup] = {st.x, st.y, st.z, st.w};
  const int col[kSyncGroup] = {me.x & 0xffff, (int)((unsigned)me.x >> 16), me.y & 0xffff,
                               (int)((unsigned)me.y >> 16)};
  const int nr = me.w;
  if (l >= me.z) return;
  T* d[kSyncGroup];
#pragma unroll
  for (int r = 0; r < kSyncGroup; ++r)
    d[r] = slot_at<T>(slots, slot[r], off[r]) + (int64_t)l * ls[r];
  T x[kSyncGroup], w[kSyncGroup][kSyncGroup];
#pragma unroll
  for (int r = 0; r < kSyncGroup; ++r) {
    x[r] = T(0);
    if (r >= nr) continue;  // no entry reads it
    load_row_weights<T>(static_cast<const T*>(s.group_w) + (r * ng + u) * kSyncGroup, w[r]);
    x[r] = *d[r];
  }
#pragma unroll
  for (int r = 0; r < kSyncGroup; ++r) {
    if (r >= nr) continue;
    T acc = T(0);
    const int n = col[r] & 7;
#pragma unroll
    for (int e = 0; e < kSyncGroup; ++e)
      if (e < n) {
        const int c = col[r] >> (3 + 2 * e);
        const T lo = c & 1 ? x[1] : x[0], hi = c & 1 ? x[3] : x[2];
        acc = fma(w[r][e], c & 2 ? hi : lo, acc);
      }
    *d[r] = acc;
  }
}

}  // namespace

cudaError_t launch_sync(int dtype, int step, const SyncCtx& s, void* const* slots,
                        const int32_t* slot_ls, cudaStream_t stream) {
  if (step == SYNC_GROUPS) {
    if (s.ngroups <= 0) return cudaSuccess;
    const int64_t n = (int64_t)s.ngroups * s.lmax;
    const int blocks = (int)((n + kGroupThreads - 1) / kGroupThreads);
    auto* k = dtype == 1 ? k_sync_groups<double> : k_sync_groups<float>;
    k<<<blocks, kGroupThreads, 0, stream>>>(s, slots);
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
