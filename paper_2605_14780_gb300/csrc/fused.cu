// Boundary conditions fused with the stencil that follows them (arxiv
// 2605.14780, Sec. IV-C: the boundary rows are only ever read by the next
// stencil, so they can be evaluated where that stencil reads them).  One
// launch over every slot computes
//
//   out[x] = sum_o c_o * f(x + o)   for every data value x,
//
// where f is the field as a forward apply leaves it: data values as stored,
// covered ghost values evaluated from their row of A and b at the point of
// use, uncovered ghost values as stored.  The same launch also writes every
// covered ghost value (f's ghosts), so the fields end as after bc_apply.
// Stencil threads never read covered ghost memory (they evaluate the row),
// so the ghost writes and the stencil reads do not race.  27-point box
// stencils with one weight off the centre take two launches instead: the
// plan's ghost fill, then k_fused_box (below) over the filled fields.
//
// Rows are the plan's level-0 rows of A in CSR form; each slot has a table
// that maps every cell of its ghost frame (the full region minus the data
// region, in slab order) to its row, or -1.  The stencil outputs go by
// tiles of 32 x 8 x 4 cells (x 1 for 2-D blocks) and one level: the CTA
// stages the tile and its halo in shared memory, evaluating each covered
// ghost of the halo once, and each thread sums the points for 4 cells
// along axis 2 from there.
#include <cstdint>

#include "bc_internal.h"

namespace bcg {
namespace {

__device__ __forceinline__ uint32_t fdivf(uint32_t n, const FastDiv& f) {
  return (__umulhi(n, f.m) + n) >> f.s;
}

template <typename T> struct FBits;
template <> struct FBits<float> { using type = uint32_t; };
template <> struct FBits<double> { using type = uint64_t; };

__device__ __forceinline__ uint32_t to_bits_f(float v) { return __float_as_uint(v); }
__device__ __forceinline__ uint64_t to_bits_f(double v) {
  return (uint64_t)__double_as_longlong(v);
}
template <typename T>
__device__ __forceinline__ T from_bits_f(typename FBits<T>::type b);
template <>
__device__ __forceinline__ float from_bits_f<float>(uint32_t b) { return __uint_as_float(b); }
template <>
__device__ __forceinline__ double from_bits_f<double>(uint64_t b) {
  return __longlong_as_double((long long)b);
}

// index of ghost cell (i, j, k) in the slot's frame table
__device__ __forceinline__ int64_t frame_index(const FuseSlot& S, int i, int j, int k) {
  const int64_t F0 = S.n[0] + 2 * S.h[0], F1 = S.n[1] + 2 * S.h[1];
  const int64_t slab = (int64_t)S.h[2] * F1 * F0;
  if (k < 0) return ((int64_t)(k + S.h[2]) * F1 + (j + S.h[1])) * F0 + (i + S.h[0]);
  if (k >= S.n[2]) return slab + ((int64_t)(k - S.n[2]) * F1 + (j + S.h[1])) * F0 + (i + S.h[0]);
  const int64_t plane = F1 * F0 - (int64_t)S.n[1] * S.n[0];
  const int64_t base = 2 * slab + (int64_t)k * plane;
  if (j < 0) return base + (int64_t)(j + S.h[1]) * F0 + (i + S.h[0]);
  if (j >= S.n[1]) return base + (int64_t)(S.h[1] + j - S.n[1]) * F0 + (i + S.h[0]);
  const int64_t b2 = base + 2 * (int64_t)S.h[1] * F0 + (int64_t)j * 2 * S.h[0];
  return i < 0 ? b2 + (i + S.h[0]) : b2 + S.h[0] + (i - S.n[0]);
}

// cell of frame entry f (the inverse of frame_index)
__device__ __forceinline__ void frame_cell(const FuseSlot& S, int64_t f, int& i, int& j, int& k) {
  const int64_t F0 = S.n[0] + 2 * S.h[0], F1 = S.n[1] + 2 * S.h[1];
  const int64_t slab = (int64_t)S.h[2] * F1 * F0;
  if (f < 2 * slab) {
    const bool top = f >= slab;
    const int64_t g = top ? f - slab : f;
    const int64_t kk = g / (F1 * F0), r = g - kk * F1 * F0;
    k = top ? S.n[2] + (int)kk : (int)kk - S.h[2];
    j = (int)(r / F0) - S.h[1];
    i = (int)(r % F0) - S.h[0];
    return;
  }
  const int64_t plane = F1 * F0 - (int64_t)S.n[1] * S.n[0];
  const int64_t g = f - 2 * slab;
  k = (int)(g / plane);
  int64_t r = g - (int64_t)k * plane;
  const int64_t band = (int64_t)S.h[1] * F0;
  if (r < 2 * band) {
    const bool top = r >= band;
    const int64_t rr = top ? r - band : r;
    j = top ? S.n[1] + (int)(rr / F0) : (int)(rr / F0) - S.h[1];
    i = (int)(rr % F0) - S.h[0];
    return;
  }
  r -= 2 * band;
  j = (int)(r / (2 * S.h[0]));
  const int t = (int)(r - (int64_t)j * 2 * S.h[0]);
  i = t < S.h[0] ? t - S.h[0] : S.n[0] + t - S.h[0];
}

__device__ __forceinline__ int64_t cell_off(const FuseSlot& S, int i, int j, int k) {
  return (int64_t)(i + S.h[0]) * S.s[0] + (int64_t)(j + S.h[1]) * S.s[1] +
         (int64_t)(k + S.h[2]) * S.s[2];
}

// row r of A at level l: bit pattern of a unit copy, else b_r + sum_e a_e x_e
template <typename T>
__device__ __forceinline__ T eval_row(const FuseCtx& F, void* const* slots, int r, int l,
                                      bool& copy, typename FBits<T>::type& bits) {
  using B = typename FBits<T>::type;
  const int e0 = __ldg(F.rptr + r), e1 = __ldg(F.rptr + r + 1);
  const T b = __ldg(static_cast<const T*>(F.rhs) + r);
  if (e1 - e0 == 1) {
    const T a = __ldg(static_cast<const T*>(F.val) + e0);
    if (a == T(1) && to_bits_f(b) == 0) {
      const int s = __ldg(F.eslot + e0);
      const B* x = static_cast<const B*>(slots[s]);
      bits = __ldg(x + (__ldg(F.eoff + e0) + (int64_t)l * __ldg(F.slot_ls + s)));
      copy = true;
      return from_bits_f<T>(bits);
    }
  }
  copy = false;
  T acc = b;
  for (int e = e0; e < e1; ++e) {
    const int s = __ldg(F.eslot + e);
    const T* x = static_cast<const T*>(slots[s]);
    acc = fma(__ldg(static_cast<const T*>(F.val) + e),
              __ldg(x + (__ldg(F.eoff + e) + (int64_t)l * __ldg(F.slot_ls + s))), acc);
  }
  return acc;
}

// f at cell (i, j, k) of slot S, level offset lo: a data value, a covered
// ghost evaluated from its row, or a stored (uncovered) ghost
template <typename T>
__device__ __forceinline__ T field_at(const FuseCtx& F, void* const* slots, const FuseSlot& S,
                                      const T* x, int i, int j, int k, int l, int64_t lo) {
  if (i >= 0 && i < S.n[0] && j >= 0 && j < S.n[1] && k >= 0 && k < S.n[2])
    return __ldg(x + (cell_off(S, i, j, k) + lo));
  const int r = __ldg(F.frame_row + S.fbase + frame_index(S, i, j, k));
  if (r < 0) return __ldg(x + (cell_off(S, i, j, k) + lo));
  bool copy;
  typename FBits<T>::type bits;
  return eval_row<T>(F, slots, r, l, copy, bits);
}

template <typename T>
__global__ void __launch_bounds__(kFuseThreads)
    k_fused(FuseCtx F, FuseStencil st, void* const* slots, void* const* outs) {
  using B = typename FBits<T>::type;
  __shared__ FuseSlot S;
  __shared__ int si;
  __shared__ T sm[kTileVals];
  __shared__ int dp[kFuseMaxPoints];
  __shared__ T cf[kFuseMaxPoints];
  const int tid = threadIdx.x;
  if (tid == 0) {
    // the slot of this CTA: the last slot whose first CTA is <= blockIdx.x
    int lo = 0, hi = F.nslots - 1;
    while (lo < hi) {
      const int mid = (lo + hi + 1) >> 1;
      if (F.slot[mid].cta0 <= (int64_t)blockIdx.x) lo = mid;
      else hi = mid - 1;
    }
    si = lo;
    S = F.slot[lo];
  }
  __syncthreads();
  const int64_t lc = (int64_t)blockIdx.x - S.cta0;
  const T* x = static_cast<const T*>(slots[si]);
  if (lc < S.tiles) {
    // stencil outputs of one tile at one level: stage the tile and its
    // halo (covered ghosts evaluated once each), then the sums
    int t = (int)lc;
    const int tx = t % S.nt[0];
    t /= S.nt[0];
    const int ty = t % S.nt[1];
    t /= S.nt[1];
    const int tzi = t % S.nt[2];
    const int l = t / S.nt[2];
    const int i0 = tx * kTileX, j0 = ty * kTileY, k0 = tzi * S.tz;
    const int SX = kTileX + 2 * st.r[0], SY = kTileY + 2 * st.r[1], SZ = S.tz + 2 * st.r[2];
    const int64_t lo = (int64_t)l * S.ls;
    for (int p = tid; p < st.n; p += kFuseThreads) {
      dp[p] = (st.o[p][2] * SY + st.o[p][1]) * SX + st.o[p][0];
      cf[p] = (T)st.c[p];
    }
    for (int e = tid; e < SX * SY * SZ; e += kFuseThreads) {
      const int li = e % SX, q = e / SX;
      const int lj = q % SY, lk = q / SY;
      const int i = i0 + li - st.r[0], j = j0 + lj - st.r[1], k = k0 + lk - st.r[2];
      const bool full = i >= -S.h[0] && i < S.n[0] + S.h[0] && j >= -S.h[1] &&
                        j < S.n[1] + S.h[1] && k >= -S.h[2] && k < S.n[2] + S.h[2];
      // cells past the full region only border outputs past the data region
      sm[e] = full ? field_at<T>(F, slots, S, x, i, j, k, l, lo) : T(0);
    }
    __syncthreads();
    const int ix = tid % kTileX, iy = tid / kTileX;
    const int i = i0 + ix, j = j0 + iy;
    if (i < S.n[0] && j < S.n[1]) {
      T* out = static_cast<T*>(outs[si]);
      for (int kz = 0; kz < S.tz; ++kz) {
        const int k = k0 + kz;
        if (k >= S.n[2]) break;
        const T* c = sm + ((kz + st.r[2]) * SY + (iy + st.r[1])) * SX + (ix + st.r[0]);
        T acc = T(0);
        for (int p = 0; p < st.n; ++p) acc = fma(cf[p], c[dp[p]], acc);
        out[cell_off(S, i, j, k) + lo] = acc;
      }
    }
    return;
  }
  // the ghost value at frame entry f, level l
  const int64_t w = (lc - S.tiles) * kFuseThreads + tid;
  if (w >= (int64_t)S.nf * S.L) return;
  B* xb = static_cast<B*>(slots[si]);
  int64_t f;
  int l;
  if (S.lfast) {
    f = (int64_t)fdivf((uint32_t)w, S.dL);
    l = (int)(w - f * S.L);
  } else {
    l = (int)fdivf((uint32_t)w, S.dnf);
    f = w - (int64_t)l * S.nf;
  }
  const int r = __ldg(F.frame_row + S.fbase + f);
  if (r < 0) return;
  int i, j, k;
  frame_cell(S, f, i, j, k);
  bool copy;
  B bits;
  const T val = eval_row<T>(F, slots, r, l, copy, bits);
  xb[cell_off(S, i, j, k) + (int64_t)l * S.ls] = copy ? bits : to_bits_f(val);
}

// Box stencils (FuseStencil::box): a x (sum over the 3 x 3 x 3 box) +
// (c0 - a) x centre.  In FP64 the general kernel is bound by the FP64 pipe
// (27 multiply-adds a value at 1.15 TFLOP/s; GB300 issues one FP64 warp
// instruction per 16 cycles and SM), so this one counts FP64 instructions:
// the box sum is taken axis by axis and neighbouring outputs share their
// pair sums (x: s = x0 + x1, rows x(-1) + s and s + x2; y and z alike),
// 1.5 adds per value and axis, 6.25 FP64 instructions per value at |a| = 1
// with 2 x 4 values a thread (2.25 for the row sums with their two halo
// rows, 1.5 + 1.5, 1 for the centre), 7.25 otherwise.  2 x 2 values a thread
// (7 instructions, twice the warps) took 8 % longer on the blocks below,
// 2 x 8 40 %, a ring of six planes with the next pair in flight 4 %.
//
// The ghosts are filled by the plan's own launch first and read from memory
// (evaluating them while staging, as the general kernel does, put chains of
// dependent loads and divergence into every tile at a face: 1107 us).  A CTA
// of 2 warps takes 32 x 16 cells (a warp 32 x 8) and walks bz planes in
// pairs; a ring of four planes with their halo sits in shared memory (20 KB
// in FP64, eight CTAs an SM: while one waits for its planes the others keep
// the pipe busy; 4 warps a CTA: 2 % longer, 1 warp: 1 %).  The sums associate
// differently from the general kernel's: against sums in higher precision they
// are the closer ones for random values (1.4e-16 to 2.2e-16 of the result's norm
// for the operator below), for smooth fields on a large mean 0.9 to 1.4 times as
// far off.  A value that is not finite is summed again in the general order from
// the ring, so infinities, NaNs and overflow come out as there.
//
// 27-point operator (26, -1), FP64, fill included: 16 blocks of 128^3 1576 -> 492
// us (6.25 instructions a value take 0.68 of the pipe's rate), one 114 -> 47,
// four of 64^3 63 -> 34, one of 16^3 even at 18 (build_fusion chooses the planes
// per tile).
__device__ __forceinline__ void cp_async_cell(double* smem, const double* gmem) {
  const unsigned sa = (unsigned)__cvta_generic_to_shared(smem);
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8;\n" ::"r"(sa), "l"(gmem) : "memory");
}

constexpr int kBoxPitch = kBoxX + 2, kBoxPlane = kBoxPitch * (kBoxY + 2);
constexpr int kBoxCtas = 512 / kBoxThreads;  // 16 warps an SM

// 3 x 3 sums of one staged plane for a thread's 2 x 4 cells; `c`: the
// staged value one row above and one cell before the thread's first
__device__ __forceinline__ void plane_sums(const double* c, double (&P)[2 * kBoxTy]) {
  double r[kBoxTy + 2][2];
#pragma unroll
  for (int j = 0; j < kBoxTy + 2; ++j) {
    const double2 a = *reinterpret_cast<const double2*>(c + j * kBoxPitch);
    const double2 b = *reinterpret_cast<const double2*>(c + j * kBoxPitch + 2);
    const double s = a.y + b.x;
    r[j][0] = a.x + s;
    r[j][1] = s + b.y;
  }
#pragma unroll
  for (int x = 0; x < 2; ++x)
#pragma unroll
    for (int j = 0; j < kBoxTy; j += 2) {
      const double s = r[j + 1][x] + r[j + 2][x];
      P[2 * j + x] = r[j][x] + s;
      P[2 * (j + 1) + x] = s + r[j + 3][x];
    }
}

// by the exponent bits: a floating compare would take the FP64 pipe
__device__ __forceinline__ bool finite_value(double v) {
  return ((unsigned)__double2hiint(v) & 0x7ff00000u) != 0x7ff00000u;
}

// v, or -v where `flip` holds the sign bit (no FP64 instruction either)
__device__ __forceinline__ double flip_sign(double v, unsigned flip) {
  return __hiloint2double((int)((unsigned)__double2hiint(v) ^ flip), __double2loint(v));
}

// UNIT: |a| = 1, a x S is S or -S
template <bool UNIT>
__global__ void __launch_bounds__(kBoxThreads, kBoxCtas)
    k_fused_box(FuseCtx F, FuseStencil st, void* const* slots, void* const* outs) {
  __shared__ FuseSlot S;
  __shared__ int si;
  __shared__ __align__(16) double ring[4][kBoxPlane];
  const int tid = threadIdx.x;
  if (tid == 0) {
    int lo = 0, hi = F.nslots - 1;  // the last slot whose first CTA is <= blockIdx.x
    while (lo < hi) {
      const int mid = (lo + hi + 1) >> 1;
      if (F.slot[mid].bcta0 <= (int64_t)blockIdx.x) lo = mid;
      else hi = mid - 1;
    }
    si = lo;
    S = F.slot[lo];
  }
  __syncthreads();
  int t = blockIdx.x - (int)S.bcta0;
  const int tx = t % S.bnt[0];
  t /= S.bnt[0];
  const int ty = t % S.bnt[1];
  t /= S.bnt[1];
  const int tz = t % S.bnt[2];
  const int l = t / S.bnt[2];
  const int i0 = tx * kBoxX, j0 = ty * kBoxY, k0 = tz * S.bz;
  const int k1 = min(k0 + S.bz, S.n[2]);
  const int warp = tid >> 5, lane = tid & 31;
  const int64_t s0 = S.s[0], s1 = S.s[1], s2 = S.s[2];
  const int64_t org = cell_off(S, i0, j0, k0) + (int64_t)l * S.ls;
  const double* x = static_cast<const double*>(slots[si]) + org;

  // planes k and k + 1 with their halo into the ring (plane k in slot k & 3),
  // a warp a row; cells past the full region only border outputs past the
  // data region and are zero
  const int iend = S.n[0] + S.h[0] - i0, jend = S.n[1] + S.h[1] - j0;
  auto stage = [&](int k) {
    for (int r = warp; r < 2 * (kBoxY + 2); r += kBoxThreads / 32) {
      const int z = r >= kBoxY + 2, j = r - z * (kBoxY + 2) - 1, kk = k + z;
      double* dst = ring[kk & 3] + (j + 1) * kBoxPitch;
      const bool row = j < jend && kk < S.n[2] + S.h[2];
      const double* src = x + ((int64_t)(kk - k0) * s2 + (int64_t)j * s1);
#pragma unroll
      for (int u = 0; u < 2; ++u) {
        const int li = lane + 32 * u;
        if (li >= kBoxPitch) break;
        if (row && li - 1 < iend)
          cp_async_cell(dst + li, src + (int64_t)(li - 1) * s0);
        else
          dst[li] = 0.0;
      }
    }
    asm volatile("cp.async.wait_all;\n" ::: "memory");
  };

  // this thread's cells: 2 along x from cx, kBoxTy along y from cy
  const int cx = 2 * (lane & 15), cy = warp * 2 * kBoxTy + (lane >> 4) * kBoxTy;
  const int at = cy * kBoxPitch + cx;  // staged value at (-1, -1) of the first cell
  // a warp whose rows all lie past the block has nothing to sum
  const bool work = j0 + warp * 2 * kBoxTy < S.n[1];
  const int nx = S.n[0] - i0 - cx, ny = S.n[1] - j0 - cy;  // this thread's cells in the block
  double* out = static_cast<double*>(outs[si]) + (org + cx * s0 + cy * s1);
  const double a = st.a, d = st.d;
  const unsigned flip = st.a < 0 ? 0x80000000u : 0u;

  // the outputs of plane k from the box sums b
  auto put = [&](int k, const double (&b)[2 * kBoxTy]) {
    const double* c = ring[k & 3] + at + kBoxPitch + 1;
    double* o = out + (int64_t)(k - k0) * s2;
#pragma unroll
    for (int j = 0; j < kBoxTy; ++j)
#pragma unroll
      for (int xx = 0; xx < 2; ++xx) {
        const double x0 = c[j * kBoxPitch + xx], s = b[2 * j + xx];
        double v = UNIT ? fma(d, x0, flip_sign(s, flip)) : fma(a, s, d * x0);
        if (!finite_value(v)) {
          v = 0.0;
          for (int p = 0; p < st.n; ++p)
            v = fma(st.c[p],
                    ring[(k + st.o[p][2]) & 3]
                        [at + (j + 1 + st.o[p][1]) * kBoxPitch + xx + 1 + st.o[p][0]],
                    v);
        }
        if (xx < nx && j < ny) o[j * s1 + xx * s0] = v;
      }
  };

  double p0[2 * kBoxTy], p1[2 * kBoxTy];  // plane sums of k - 1 and k
  stage(k0 - 1);
  __syncthreads();
  if (work) {
    plane_sums(ring[(k0 - 1) & 3] + at, p0);
    plane_sums(ring[k0 & 3] + at, p1);
  }
  for (int k = k0; k < k1; k += 2) {
    stage(k + 1);
    __syncthreads();
    if (work) {
      double p2[2 * kBoxTy], b[2 * kBoxTy];
      plane_sums(ring[(k + 1) & 3] + at, p2);
#pragma unroll
      for (int q = 0; q < 2 * kBoxTy; ++q) {
        p1[q] += p2[q];         // planes k and k + 1, shared by both outputs
        b[q] = p0[q] + p1[q];
        p0[q] = p2[q];
      }
      put(k, b);
      if (k + 1 < k1) {
        plane_sums(ring[(k + 2) & 3] + at, p2);
#pragma unroll
        for (int q = 0; q < 2 * kBoxTy; ++q) {
          b[q] = p1[q] + p2[q];
          p1[q] = p2[q];
        }
        put(k + 1, b);
      }
    }
    __syncthreads();  // planes k - 1 and k are free for k + 3 and k + 4
  }
}

}  // namespace

cudaError_t launch_fused(int dtype, const FuseCtx& F, const FuseStencil& st, void* const* slots,
                         void* const* outs, int64_t nctas, cudaStream_t s) {
  if (nctas <= 0) return cudaSuccess;
  if (dtype == 1)
    k_fused<double><<<(unsigned)nctas, kFuseThreads, 0, s>>>(F, st, slots, outs);
  else
    k_fused<float><<<(unsigned)nctas, kFuseThreads, 0, s>>>(F, st, slots, outs);
  return cudaGetLastError();
}

cudaError_t launch_fused_box(const FuseCtx& F, const FuseStencil& st, void* const* slots,
                             void* const* outs, int64_t nctas, cudaStream_t s) {
  if (nctas <= 0) return cudaSuccess;
  const bool unit = st.a == 1.0 || st.a == -1.0;
  auto* kernel = unit ? k_fused_box<true> : k_fused_box<false>;
  kernel<<<(unsigned)nctas, kBoxThreads, 0, s>>>(F, st, slots, outs);
  return cudaGetLastError();
}

}  // namespace bcg
