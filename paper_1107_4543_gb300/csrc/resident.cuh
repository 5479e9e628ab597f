// Batched step for small lattices held in shared memory for all the time
// steps of one launch (section 2.1, Eq. blbs, as the per-step kernels): one
// thread block per member loads the member's nine planes into shared memory,
// runs its n steps there and writes the result back once: its 9 x nx ny
// elements cross HBM once in and once out for the whole launch instead of in
// and out at every step.
//
// The steps work in place (the "AA" access pattern of Bailey, Myre, Walsh,
// Lilja and Saar, ICPP 2009): even steps pull population i of node x from
// slot (i, x - c_i) and put the post-collision population of the opposite
// direction there, so that odd steps find what streams to node x in its own
// slots, each in the slot of the opposite direction, and leave the
// post-collision populations in their own.  Every slot is read and written
// by one node per step, so one set of planes is enough where a second buffer
// had left most members alone on their SM: two members per SM now hide each
// other's latency and barriers.
//
// The arithmetic is the per-step kernels' own (collide_pair_hl, the packed
// form of collide_dev, for FP32, collide_pair for the 16-bit types, the same
// storage rounding), node by node, so a member's result is bit-identical to
// the per-step path's.
#pragma once
#include <type_traits>

#include "bounds.cuh"
#include "lbm_internal.h"
#include "step_multi.cuh"

namespace lbm {

// 384 threads (12 warps) per member, two blocks per SM at the 80-register
// cap, no spills: 1,024 lattices of 32^2 - 56^2 take 4.8 ms for 500 steps
// (512 threads at 64 registers, 100 bytes of spills: 6.5; 320: 5.2; two step
// buffers, one node per thread, 512 threads: 7.65)
constexpr int kResidentThreads = 384;

template <typename T>
__device__ __forceinline__ uint32_t bits16(const T *p) {
  return (uint32_t) * reinterpret_cast<const unsigned short *>(p);
}

__device__ constexpr int opposite(int i) {
  return i == 0 ? 0 : (i <= 2 ? i + 2 : (i <= 4 ? i - 2 : (i <= 6 ? i + 2 : i - 2)));
}

// (x, y) of item r, advanced by a fixed stride of (dx, dy) = (stride mod nx,
// stride / nx) without a division per item
struct Walk {
  int x, y, dx, dy, nx;
  __device__ __forceinline__ Walk(int r, int stride, int nx_) : nx(nx_) {
    y = r / nx;
    x = r - y * nx;
    dy = stride / nx;
    dx = stride - dy * nx;
  }
  __device__ __forceinline__ void next() {
    x += dx;
    y += dy;
    if (x >= nx) {
      x -= nx;
      ++y;
    }
  }
};

// Node (x, y) and the slots that the directions pull from, periodic
struct Nbr {
  int r0;          // y nx
  int xm, x, xp;   // x - 1, x, x + 1 (wrapped)
  int ym, yp;      // (y - 1) nx, (y + 1) nx (wrapped)
  __device__ __forceinline__ int at(int i) const {
    const int cx = CXd(i), cy = CYd(i);
    return (cy == 1 ? ym : (cy == -1 ? yp : r0)) + (cx == 1 ? xm : (cx == -1 ? xp : x));
  }
};
__device__ __forceinline__ Nbr nbr(int x, int y, int nx, int ny) {
  Nbr n;
  n.x = x;
  n.r0 = y * nx;
  n.xm = x == 0 ? nx - 1 : x - 1;
  n.xp = x == nx - 1 ? 0 : x + 1;
  n.ym = (y == 0 ? ny - 1 : y - 1) * nx;
  n.yp = (y == ny - 1 ? 0 : y + 1) * nx;
  return n;
}

// the collision constants, behind the planes
template <typename T> struct ResidentConst;
template <> struct ResidentConst<float> {
  using Table = HlPairs;
  static constexpr int COUNT = HL_COUNT;
  static __device__ __forceinline__ float value(const DevParams &P, int k) { return hl_const(P, k); }
  static __device__ __forceinline__ const HlPairs &of(const Table &t) { return t; }
};
template <typename T> struct ResidentConst {
  struct alignas(16) Table {
    float2 c[PC_COUNT];
  };
  static constexpr int COUNT = PC_COUNT;
  static __device__ __forceinline__ float value(const DevParams &P, int k) {
    return pair_const(P, k);
  }
  static __device__ __forceinline__ SharedPairs of(const Table &t) { return SharedPairs{t.c}; }
};

// Slots (ia, ib) of the planes as the two nodes of a pair
template <typename T>
__device__ __forceinline__ F2 slot_load(const T *A, int ia, int ib) {
  if constexpr (sizeof(T) == 4) {
    return f2(A[ia], A[ib]);
  } else {
    float u[2];
    Elem<T>::unpack2(bits16(A + ia) | bits16(A + ib) << 16, u);
    return f2(u[0], u[1]);
  }
}
template <typename T>
__device__ __forceinline__ void slot_store(T *A, int ia, int ib, bool two, F2 f) {
  float u, v;
  f2split(f, u, v);
  if constexpr (sizeof(T) == 4) {
    A[ia] = u;
    if (two) A[ib] = v;
  } else {
    const uint32_t w = Elem<T>::pack2(u, v);
    reinterpret_cast<unsigned short *>(A)[ia] = (unsigned short)(w & 0xffffu);
    if (two) reinterpret_cast<unsigned short *>(A)[ib] = (unsigned short)(w >> 16);
  }
}

// The member's nine planes into shared memory, and back after n steps: a
// node's nine elements at a time, so that nine loads are in flight and share
// one address computation.  us per call of one step, one element of one plane
// at a time (with its divisions) / nine: four FP16 members of 80^2 107 / 28, of
// 2 x 3000 131 / 85, FP32 of 55 x 56 64 / 22.
template <typename T>
__device__ __forceinline__ void resident_load(T *A, const T *__restrict__ src, const Geom &g, int N) {
  Walk w(threadIdx.x, blockDim.x, g.nx);
  for (int r = threadIdx.x; r < N; r += blockDim.x, w.next()) {
    const T *p = src + (long long)bounds::ck(w.y, g.ny, bounds::RES_NODE) * g.rstride + w.x;
    T v[9];
#pragma unroll
    for (int i = 0; i < 9; ++i) v[i] = p[(long long)i * g.plane];
#pragma unroll
    for (int i = 0; i < 9; ++i) A[i * N + r] = v[i];
  }
}
template <typename T>
__device__ __forceinline__ void resident_store(const T *A, T *__restrict__ dst, const Geom &g, int N,
                                               int n) {
  Walk w(threadIdx.x, blockDim.x, g.nx);
  for (int r = threadIdx.x; r < N; r += blockDim.x, w.next()) {
    T *p = dst + (long long)bounds::ck(w.y, g.ny, bounds::RES_NODE) * g.rstride + w.x;
    if (n & 1) {  // post-collision population i of x is in slot (opposite i, x + c_i)
      const Nbr b = nbr(w.x, w.y, g.nx, g.ny);
#pragma unroll
      for (int i = 0; i < 9; ++i)
        p[(long long)i * g.plane] = A[opposite(i) * N + b.at(opposite(i))];
    } else {
#pragma unroll
      for (int i = 0; i < 9; ++i) p[(long long)i * g.plane] = A[i * N + r];
    }
  }
}

// idx[b]: the entry block b steps.  Each member takes min(steps, limits[e])
// steps (limits may be null) from buffer parity ^ off and leaves its state
// in the buffer that parity of steps selects, as the per-step launches do.
//
// A thread takes two nodes at a time for the packed collisions: node p and
// node p + ceil(N / 2) of the row-major order, so that a warp's accesses to
// either are consecutive words whatever the row length (adjacent nodes would
// hit every bank twice, half rows apart a warp spans rows and does so too:
// 37% of the shared-memory wavefronts, which bound the kernel, were
// conflicts).
template <typename T>
__global__ void __launch_bounds__(kResidentThreads, 2)
k_batch_resident(const BatchEntry *__restrict__ ents, const int *__restrict__ idx, int nents,
                 int parity, int steps, const int *__restrict__ limits, int consts_at) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int e = idx[blockIdx.x];
  if (!bounds::ok(e >= 0 && e < nents, bounds::BATCH_REC)) return;  // block-uniform
  const BatchEntry &E = ents[e];
  const int nx = E.g.nx, ny = E.g.ny, N = nx * ny;
  if (!bounds::ok(9 * N * (int)sizeof(T) <= consts_at, bounds::RES_NODE)) return;  // block-uniform
  int n = steps;
  if (limits != nullptr && limits[e] < n) n = limits[e];
  if (n <= 0) return;  // block-uniform
  const int from = parity ^ E.off;
  const T *src = static_cast<const T *>(E.buf[from]);
  T *A = reinterpret_cast<T *>(smem_raw);
  using RC = ResidentConst<T>;
  typename RC::Table &table = *reinterpret_cast<typename RC::Table *>(smem_raw + consts_at);
  resident_load(A, src, E.g, N);
  if (threadIdx.x < RC::COUNT) {
    // thread k's constant.  FP32 reads all of them at once; the 16 of the other
    // types, each thread its own, cost 1 us more in a launch but leave the
    // step loop better scheduled: four FP16 members of 80^2 4.74 instead of
    // 4.91 us per step
    float v = 0.0f;
    if constexpr (sizeof(T) == 4) {
#pragma unroll
      for (int k = 0; k < RC::COUNT; ++k) {
        const float c = RC::value(E.dp, k);
        if (threadIdx.x == k) v = c;
      }
    } else {
      v = RC::value(E.dp, threadIdx.x);
    }
    table.c[threadIdx.x] = make_float2(v, v);
  }
  __syncthreads();
  const int half = (N + 1) >> 1;
  for (int t = 0; t < n; ++t) {
    if (!(t & 1)) {
      Walk wa(threadIdx.x, blockDim.x, nx), wb(threadIdx.x + half, blockDim.x, nx);
      for (int p = threadIdx.x; p < half; p += blockDim.x, wa.next(), wb.next()) {
        // an odd lattice's last pair is one node (taken twice, stored once)
        const bool two = p + half < N;
        const Nbr a = nbr(wa.x, bounds::ck(wa.y, ny, bounds::RES_NODE), nx, ny);
        const Nbr b = two ? nbr(wb.x, bounds::ck(wb.y, ny, bounds::RES_NODE), nx, ny) : a;
        F2 f[9];
#pragma unroll
        for (int i = 0; i < 9; ++i) f[i] = slot_load(A, i * N + a.at(i), i * N + b.at(i));
        collide_two<T>(f, RC::of(table));
#pragma unroll
        for (int i = 0; i < 9; ++i)
          slot_store(A, i * N + a.at(i), i * N + b.at(i), two, f[opposite(i)]);
      }
    } else {
      for (int p = threadIdx.x; p < half; p += blockDim.x) {
        const bool two = p + half < N;
        const int q = two ? p + half : p;
        F2 f[9];
#pragma unroll
        for (int i = 0; i < 9; ++i) f[opposite(i)] = slot_load(A, i * N + p, i * N + q);
        collide_two<T>(f, RC::of(table));
#pragma unroll
        for (int i = 0; i < 9; ++i) slot_store(A, i * N + p, i * N + q, two, f[i]);
      }
    }
    __syncthreads();
  }
  // the entry anew: its geometry and pointers would hold registers in the loop
  // (8 bytes of spills, 4.91 us per step of four FP16 members of 80^2)
  const BatchEntry *F = ents + e;
  asm volatile("" : "+l"(F));
  resident_store(A, static_cast<T *>(F->buf[from ^ (n & 1)]), F->g, N, n);
}

// FP32 members of at most kResidentScalar nodes, the same pattern with one
// node per thread: so few nodes leave lanes idle in pairs, and a step is one
// chain of shared-memory reads, collision and barrier, which the scalar
// collision, its constants in registers, makes shorter; blocks as small as
// the members let several share an SM.  us per step, in pairs by
// k_batch_resident / here, 100 members: 3^2 0.41 / 0.22, 10^2 0.41 / 0.24, 16^2
// 0.41 / 0.30, 18^2 0.55 / 0.40; 600 members: 16^2 1.02 / 0.84, 18^2 1.67 /
// 1.26.  (Two step buffers, one node per thread, 512 threads for every size:
// 0.28, 0.29, 0.40, 0.53; 1.28, 1.81.)
static __global__ void __launch_bounds__(kResidentScalar)
k_resident_tiny(const BatchEntry *__restrict__ ents, const int *__restrict__ idx, int nents,
                int parity, int steps, const int *__restrict__ limits) {
  __shared__ float A[9 * kResidentScalar];
  const int e = idx[blockIdx.x];
  if (!bounds::ok(e >= 0 && e < nents, bounds::BATCH_REC)) return;  // block-uniform
  const BatchEntry &E = ents[e];
  const int nx = E.g.nx, ny = E.g.ny, N = nx * ny;
  if (!bounds::ok(N <= (int)blockDim.x, bounds::RES_NODE)) return;
  int n = steps;
  if (limits != nullptr && limits[e] < n) n = limits[e];
  if (n <= 0) return;  // block-uniform
  const int from = parity ^ E.off, r = threadIdx.x;
  resident_load(A, static_cast<const float *>(E.buf[from]), E.g, N);
  const Nbr nb = nbr(r % nx, r / nx, nx, ny);
  for (int t = 0; t < n; ++t) {
    __syncthreads();
    float f[9];
    if (r < N && !(t & 1)) {
#pragma unroll
      for (int i = 0; i < 9; ++i) f[i] = A[i * N + nb.at(i)];
      collide_dev<true, false>(f[0], f[1], f[2], f[3], f[4], f[5], f[6], f[7], f[8], E.dp);
#pragma unroll
      for (int i = 0; i < 9; ++i) A[i * N + nb.at(i)] = f[opposite(i)];
    } else if (r < N) {
#pragma unroll
      for (int i = 0; i < 9; ++i) f[opposite(i)] = A[i * N + r];
      collide_dev<true, false>(f[0], f[1], f[2], f[3], f[4], f[5], f[6], f[7], f[8], E.dp);
#pragma unroll
      for (int i = 0; i < 9; ++i) A[i * N + r] = f[i];
    }
  }
  __syncthreads();
  resident_store(A, static_cast<float *>(E.buf[from ^ (n & 1)]), E.g, N, n);
}

// nodes: those of the largest member of the launch
template <typename T>
cudaError_t launch_resident_t(const BatchEntry *ents, const int *idx, int nres, int nents,
                              long long nodes, int parity, long steps, const int *limits,
                              cudaStream_t st) {
  if (nres < 1 || steps < 1) return cudaSuccess;
  constexpr size_t table = resident_table((int)sizeof(T));
  static_assert(table == sizeof(typename ResidentConst<T>::Table) && table % 16 == 0, "table bytes");
  const size_t smem = resident_smem(nodes, (int)sizeof(T)), at = smem - table;
  cudaError_t e = cudaFuncSetAttribute(
      k_batch_resident<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, kMaxSmem);
  if (e != cudaSuccess) return e;
  // launches of at most 2^30 steps (the step count is an int on the device)
  const long chunk = 1L << 30;
  for (long done = 0; done < steps; done += chunk) {
    const long k = steps - done < chunk ? steps - done : chunk;
    bool tiny = false;
    if constexpr (sizeof(T) == 4) {
      tiny = nodes <= kResidentScalar;
      if (tiny)
        k_resident_tiny<<<(unsigned)nres, (unsigned)(nodes + 31) / 32 * 32, 0, st>>>(
            ents, idx, nents, parity ^ (int)(done & 1), (int)k, limits);
    }
    if (!tiny)
      k_batch_resident<T><<<(unsigned)nres, kResidentThreads, smem, st>>>(
          ents, idx, nents, parity ^ (int)(done & 1), (int)k, limits, (int)at);
    e = cudaGetLastError();
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

}  // namespace lbm
