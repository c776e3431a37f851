// Packing of block boxes into one contiguous buffer, for the exchange of
// ghost sources between processes that own different blocks (arxiv
// 2605.14780, Sec. V-B: each process receives the bounding box of the
// remote data its boundary rows read).  A box is a cell range of one block,
// taken with every component and level; in the buffer it is stored
// [component][level][k][j][i], boxes back to back.
//
// The copy is bound by its latency chain and by the transposition where the
// levels are contiguous in the field but the cells in the buffer.  A CTA
// takes a tile of up to 2048 values (cells x levels of one component); its
// {box, component, first cell, first level} is looked up, not searched, and
// the element offsets of the tile's cells are worked out once into shared
// memory.  Levels contiguous in the field: the tile is read levels fastest
// (runs of the field) and written cells fastest (runs of the buffer) through
// shared memory; otherwise both sides run over the cells and the tile goes
// through registers.  Strips of 128 blocks, 25.8 MB moved, levels
// innermost: 14.3 us (one value a thread, the box found by one thread's
// binary search while 255 wait, reads strided by the level count: 45.0 us).
#include <cstdint>

#include "bc_internal.h"

namespace bcg {
namespace {

__device__ __forceinline__ uint32_t pdiv(uint32_t n, const FastDiv& f) {
  return (__umulhi(n, f.m) + n) >> f.s;
}

constexpr int kPackUnroll = 4;  // values in flight per thread

template <typename B>
__global__ void __launch_bounds__(kPackThreads)
    k_pack(const PackBox* __restrict__ boxes, const int4* __restrict__ tiles, void* const* slots,
           B* buf) {
  __shared__ PackBox bx;
  __shared__ int64_t coff[kPackCells];
  __shared__ B sm[kPackVals + kPackLevels];
  constexpr int U = kPackUnroll, W = kPackThreads;
  const int tid = threadIdx.x;
  const int4 t = __ldg(tiles + blockIdx.x);  // {box, component, first cell, first level}
  if (tid < (int)(sizeof(PackBox) / 4))
    reinterpret_cast<int*>(&bx)[tid] = __ldg(reinterpret_cast<const int*>(boxes + t.x) + tid);
  __syncthreads();
  const int nc = bx.nc, nl = bx.nl;
  const int cells = min(nc, bx.cells - t.z), levels = min(nl, bx.L - t.w);
  for (int m = tid; m < cells; m += W) {
    const uint32_t q = (uint32_t)(t.z + m);
    const uint32_t row = pdiv(q, bx.d0), k = pdiv(row, bx.d1);
    const int i = (int)(q - row * (uint32_t)bx.e[0]), j = (int)(row - k * (uint32_t)bx.e[1]);
    coff[m] = (int64_t)(bx.lo[0] + i) * bx.s[0] + (int64_t)(bx.lo[1] + j) * bx.s[1] +
              (int64_t)(bx.lo[2] + (int)k) * bx.s[2];
  }
  __syncthreads();
  const B* src = static_cast<const B*>(slots[bx.slot0 + t.y]) + (int64_t)t.w * bx.ls;
  B* dst = buf + (bx.dst + ((int64_t)t.y * bx.L + t.w) * bx.cells + t.z);
  const int total = nc * nl;
  if (bx.lfast) {
    const int pitch = nc | 1;  // odd: a column of levels lies in distinct banks
    for (int f0 = tid; f0 < total; f0 += W * U) {
      B v[U];
      int at[U];
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const int f = f0 + W * u, m = (int)pdiv((uint32_t)f, bx.dnl), l = f - m * nl;
        at[u] = m < cells && l < levels ? l * pitch + m : -1;
        if (at[u] >= 0) v[u] = __ldg(src + (coff[m] + l));
      }
#pragma unroll
      for (int u = 0; u < U; ++u)
        if (at[u] >= 0) sm[at[u]] = v[u];
    }
    __syncthreads();
    for (int f = tid; f < total; f += W) {
      const int l = (int)pdiv((uint32_t)f, bx.dnc), m = f - l * nc;
      if (m < cells && l < levels) dst[(int64_t)l * bx.cells + m] = sm[l * pitch + m];
    }
  } else {
    for (int f0 = tid; f0 < total; f0 += W * U) {
      B v[U];
      int64_t at[U];
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const int f = f0 + W * u, l = (int)pdiv((uint32_t)f, bx.dnc), m = f - l * nc;
        at[u] = m < cells && l < levels ? (int64_t)l * bx.cells + m : -1;
        if (at[u] >= 0) v[u] = __ldg(src + (coff[m] + l * bx.ls));
      }
#pragma unroll
      for (int u = 0; u < U; ++u)
        if (at[u] >= 0) dst[at[u]] = v[u];
    }
  }
}

}  // namespace

cudaError_t launch_pack(int esize, const PackBox* boxes, const int4* tiles, int64_t ntiles,
                        void* const* slots, void* buf, cudaStream_t s) {
  if (ntiles <= 0) return cudaSuccess;
  if (esize == 8)
    k_pack<uint64_t><<<(unsigned)ntiles, kPackThreads, 0, s>>>(boxes, tiles, slots,
                                                                static_cast<uint64_t*>(buf));
  else
    k_pack<uint32_t><<<(unsigned)ntiles, kPackThreads, 0, s>>>(boxes, tiles, slots,
                                                                static_cast<uint32_t*>(buf));
  return cudaGetLastError();
}

}  // namespace bcg
