// Several time steps of section 2.1 (Eq. blbs) per launch, for the 32- and
// 16-bit deviation storage types: the arithmetic is the single-step
// kernels' own, node by node and step by step, with the storage rounding
// between the steps, so results are bit-identical to single steps.
//
// A single step moves 9 reads and 9 writes of one stored population per
// node (72 B in FP32, 36 B in 16 bits) for ~100 FP32 operations, so one
// lattice larger than the L2 was bound by HBM at 7.2 TB/s (99 GLUPS FP32)
// with the FMA pipe a third busy, and one of 10^4 nodes by the ~2.4 us of a
// launch.  Both kernels here trade a halo of redundant nodes for fewer
// passes over memory and fewer launches:
//
//   k_step_rows  (large lattices, batches): each warp marches along y over
//     30 chunks of kRowsV nodes, kRowSteps time levels deep; level l of row y
//     needs level l-1 of rows y-1, y, y+1, which the warp has just computed,
//     so intermediate levels live in lane-private shared-memory slots and no
//     warp waits for another.
//   k_step_tile  (small lattices): each block loads a tile with a halo as
//     wide as the steps of the launch into shared memory and steps it there,
//     the valid part shrinking by one node per side and step.
#pragma once
#include <type_traits>

#include "bounds.cuh"
#include "lbm_internal.h"
#include "pdl.cuh"

namespace lbm {

// collision constants of a storage type as a kernel parameter
template <typename T> struct PairParams { using type = DevParams; };
template <> struct PairParams<float> { using type = HlPairs; };

template <typename T>
inline typename PairParams<T>::type pair_params(const DevParams &P) {
  if constexpr (sizeof(T) == 4) return hl_pairs(P);
  else return P;
}

// 16-bit constants as broadcast pairs in shared memory (PairConst order)
struct SharedPairs {
  static constexpr bool kTable = false;
  const float2 *c;  // 16-byte aligned
  __device__ __forceinline__ F2x2 two(PairConst k) const {
    const float4 v = *reinterpret_cast<const float4 *>(c + k);
    return {f2(v.x, v.y), f2(v.z, v.w)};
  }
};

// two nodes of a storage type (the FP32 values, or the unpacked 16-bit ones)
template <typename T, typename K>
__device__ __forceinline__ void collide_two(F2 (&f)[9], const K &P) {
  if constexpr (sizeof(T) == 4)
    collide_pair_hl(f[0], f[1], f[2], f[3], f[4], f[5], f[6], f[7], f[8], P);
  else
    collide_pair<std::is_same<T, __half>::value>(f[0], f[1], f[2], f[3], f[4], f[5], f[6], f[7],
                                                 f[8], P);
}

// ------------------------------------------------------------------ rows
// The end of a row whose last chunk is partial: that chunk's lane hands its
// last real node, element el, to the next lane (chunk 0) and takes that
// lane's node 0 after it.  `warp`: some lane of the warp holds such a chunk
// (warp-uniform, so the other warps skip the selects).
template <int W>
struct Seam {
  bool warp, last;
  int el;
  // all ones for this lane's word that holds element el (a comparison per
  // word instead is turned into an indexed array in local memory, at half
  // the speed), and the shift that brings a 16-bit el to the word's high half
  uint32_t word[W];
  int up;
};

// One lane's chunk of a plane (kRowsV nodes in W words) shifted by the x
// component of the plane's velocity: the missing element comes from the
// neighbouring lane, whose chunk is the neighbouring one.
template <typename T, int W>
__device__ __forceinline__ void shift_chunk(uint32_t (&w)[W], int cx, const Seam<W> &S) {
  if (cx == 1) {
    uint32_t tail = w[W - 1];
    if (S.warp) {
      uint32_t own = 0, any = 0;
#pragma unroll
      for (int q = 0; q < W; ++q) {
        own |= w[q] & S.word[q];
        any |= S.word[q];
      }
      tail = ((tail & ~any) | own) << S.up;
    }
    const uint32_t prev = __shfl_up_sync(0xffffffffu, tail, 1);
#pragma unroll
    for (int q = W - 1; q >= 0; --q) {
      const uint32_t before = q > 0 ? w[q > 0 ? q - 1 : 0] : prev;
      w[q] = sizeof(T) == 4 ? before : __byte_perm(before, w[q], 0x5432);
    }
  } else if (cx == -1) {
    const uint32_t next = __shfl_down_sync(0xffffffffu, w[0], 1);
#pragma unroll
    for (int q = 0; q < W; ++q) {
      const uint32_t after = q < W - 1 ? w[q < W - 1 ? q + 1 : 0] : next;
      w[q] = sizeof(T) == 4 ? after : __byte_perm(w[q], after, 0x5432);
    }
    if (S.warp) {
      // node 0 takes the element after the last one
      uint32_t keep = 0, put = next;
      if constexpr (sizeof(T) == 2) {
        keep = (S.el & 1) ? 0xffffu : 0xffff0000u;
        put = (S.el & 1) ? next << 16 : next & 0xffffu;
      }
#pragma unroll
      for (int q = 0; q < W; ++q) {
        const uint32_t m = S.word[q] & ~keep;
        w[q] = (w[q] & ~m) | (put & m);
      }
    }
  }
}

// all nodes of a lane's chunk, two at a time
template <typename T, int W, typename K>
__device__ __forceinline__ void collide_chunk(uint32_t (&w)[9][W], const K &P) {
#pragma unroll
  for (int k = 0; k < kRowsV / 2; ++k) {
    F2 f[9];
#pragma unroll
    for (int i = 0; i < 9; ++i) {
      if constexpr (sizeof(T) == 4) {
        f[i] = f2(__uint_as_float(w[i][2 * k]), __uint_as_float(w[i][2 * k + 1]));
      } else {
        float t[2];
        Elem<T>::unpack2(w[i][k], t);
        f[i] = f2(t[0], t[1]);
      }
    }
    collide_two<T>(f, P);
#pragma unroll
    for (int i = 0; i < 9; ++i) {
      float a, b;
      f2split(f[i], a, b);
      if constexpr (sizeof(T) == 4) {
        w[i][2 * k] = __float_as_uint(a);
        w[i][2 * k + 1] = __float_as_uint(b);
      } else {
        w[i][k] = Elem<T>::pack2(a, b);
      }
    }
  }
}

// a lane's chunk in memory
template <typename T> struct RowsVec { using type = uint2; };
template <> struct RowsVec<float> { using type = uint4; };
__device__ __forceinline__ void set_words(uint32_t (&w)[4], const uint4 &v) {
  w[0] = v.x; w[1] = v.y; w[2] = v.z; w[3] = v.w;
}
__device__ __forceinline__ void set_words(uint32_t (&w)[2], const uint2 &v) {
  w[0] = v.x; w[1] = v.y;
}
__device__ __forceinline__ uint4 get_words(const uint32_t (&w)[4]) {
  return make_uint4(w[0], w[1], w[2], w[3]);
}
__device__ __forceinline__ uint2 get_words(const uint32_t (&w)[2]) { return make_uint2(w[0], w[1]); }

__device__ __forceinline__ void cp_async(uint4 *smem, const void *g) {
  const unsigned a = (unsigned)__cvta_generic_to_shared(smem);
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(a), "l"(g) : "memory");
}
__device__ __forceinline__ void cp_async(uint2 *smem, const void *g) {
  const unsigned a = (unsigned)__cvta_generic_to_shared(smem);
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(a), "l"(g) : "memory");
}
// shared memory of one warp of k_step_rows, in chunks: 9 incoming ones and,
// per level boundary, 3 delayed by one row and 3 by two rows, for 32 lanes
constexpr int rows_smem_chunks(int steps) { return (9 + 9 * (steps - 1)) * 32; }

// The lattice's rows are cut into segments of rg.rows; a segment is a
// sequence of halo + nchunks + halo lane positions (the chunks before chunk
// 0, chunks 0 .. nchunks - 1, those after the last, taken periodically), the
// segments' sequences follow one another, and task t takes the 32 positions
// from (32 - 2 halo) t: its middle lanes advance their chunks, each with its
// neighbours in the neighbouring lanes, and a warp spans segments freely.
// (Strips of whole warps left 20% of the lanes of the 128-lattice FP32 sweep
// idle and 27% in FP16.)  halo is 1 lane, or 2 where a partial last chunk
// has fewer nodes than the launch has steps.  (Making the chunks around the
// end of such a row whole instead, by element-wise copies or by assembling
// two aligned chunks, cost 25 - 35% of the rate of ragged FP32 lattices.)
//
// After each level one more node of each halo chunk is invalid, so STEPS <=
// kRowsV levels leave the own chunks exact; in y each level loses one row per
// side, so level l (1 .. STEPS) covers rows y0 - (STEPS - l) .. y1 - 1 +
// (STEPS - l).  In iteration j level 1 takes row y0 - (STEPS - 1) + j and
// level l the row l - 1 below it: its populations with c_y = -1 come from
// the row just computed (registers), those with c_y = 0 from the iteration
// before and those with c_y = +1 from two before (the delay slots, which
// only this lane touches: no synchronization).  The next incoming row is copied to
// shared memory (cp.async) as soon as this one's values have been shifted --
// consumed, so the lane's own slots are free -- and no register holds a load
// in flight: with the loads in registers the compiler spilled (FP32 152
// bytes at 168 registers) and the two-step form ran at 125 instead of 174
// GLUPS.
//
template <typename T, int STEPS, typename K>
__device__ __forceinline__ void rows_task(const T *__restrict__ src, T *__restrict__ dst,
                                          const Geom &g, const RowsGeom &rg, const K &par,
                                          unsigned task, int lane, typename RowsVec<T>::type *sm) {
  constexpr int V = kRowsV, W = V * (int)sizeof(T) / 4;
  using Vec = typename RowsVec<T>::type;
  static_assert(STEPS >= 2 && STEPS <= V, "the halo chunk covers V nodes");
  const int H = rg.halo, nchunks = rows_chunks(g);
  const unsigned per = (unsigned)(nchunks + 2 * H);
  const unsigned pos = task * (unsigned)(32 - 2 * H) + (unsigned)lane;
  unsigned seg = pos / per;
  const int vc = (int)(pos - seg * per) - H;  // chunk before the wrap
  const bool in = seg < (unsigned)rg.segs;
  if (!in) seg = 0;
  const bool out = in && lane >= H && lane < 32 - H && vc >= 0 && vc < nchunks;
  const int y0 = (int)seg * rg.rows, y1 = min(y0 + rg.rows, g.ny);
  const int c = bounds::ck(vc < 0 ? vc + nchunks : (vc >= nchunks ? vc - nchunks : vc), nchunks,
                           bounds::ROWS_NODE);
  const int x0 = c * V;
  Seam<W> S;
  S.el = (g.nx - 1) & (V - 1);
  S.last = c == nchunks - 1;
  S.warp = S.el != V - 1 && __any_sync(0xffffffffu, S.last);
#pragma unroll
  for (int q = 0; q < W; ++q)
    S.word[q] = S.last && S.el * (int)sizeof(T) / 4 == q ? 0xffffffffu : 0u;
  S.up = sizeof(T) == 2 && S.last && !(S.el & 1) ? 16 : 0;
  const int ya = y0 - (STEPS - 1);
  const int n = rg.rows + 2 * (STEPS - 1);
  auto row_of = [&](int y) -> const T * {
    while (y < 0) y += g.ny;
    while (y >= g.ny) y -= g.ny;
    return src + (long long)bounds::ck(y, g.ny, bounds::ROWS_NODE) * g.rstride;
  };
  Vec *raw = sm + lane, *dly = sm + 9 * 32 + lane;
  const T *pm = row_of(ya - 1) + x0, *pc = row_of(ya) + x0, *pp = row_of(ya + 1) + x0;
  int fetched = 0;
  auto fetch = [&]() {  // level 1's row ya + fetched
    if (fetched < n) {
#pragma unroll
      for (int i = 0; i < 9; ++i) {
        const T *row = CYd(i) == 1 ? pm : (CYd(i) == -1 ? pp : pc);
        cp_async(raw + i * 32, row + (long long)i * g.plane);
      }
      ++fetched;
      pm = pc;
      pc = pp;
      pp = row_of(ya + 1 + fetched) + x0;
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  fetch();
  T *drow = dst + (long long)y0 * g.rstride + x0;
  // padding chunks that complete the row's last sector (see fills_sector)
  constexpr int SECTOR = 32 / (int)sizeof(Vec);
  const int fill = out && S.last ? (SECTOR - nchunks % SECTOR) % SECTOR : 0;
  for (int j = 0; j < n; ++j) {
    asm volatile("cp.async.wait_group 0;" ::: "memory");
    uint32_t w[9][W];
#pragma unroll
    for (int i = 0; i < 9; ++i) set_words(w[i], raw[i * 32]);
#pragma unroll
    for (int i = 0; i < 9; ++i) shift_chunk<T, W>(w[i], CXd(i), S);
    fetch();
    collide_chunk<T, W>(w, par);
#pragma unroll
    for (int l = 1; l < STEPS; ++l) {
      if (j < 2 * (l - 1)) break;  // level l has no row yet
      Vec *a = dly + (l - 1) * (9 * 32), *b = a + (3 + 3 * (j & 1)) * 32;
      uint32_t u[9][W];
      set_words(u[0], a[0]); set_words(u[1], a[32]); set_words(u[3], a[64]);
      set_words(u[2], b[0]); set_words(u[5], b[32]); set_words(u[6], b[64]);
      a[0] = get_words(w[0]); a[32] = get_words(w[1]); a[64] = get_words(w[3]);
      b[0] = get_words(w[2]); b[32] = get_words(w[5]); b[64] = get_words(w[6]);
      if (j < 2 * l) break;
#pragma unroll
      for (int i = 0; i < 9; ++i) {
        if (CYd(i) != -1) {
#pragma unroll
          for (int q = 0; q < W; ++q) w[i][q] = u[i][q];
        }
        shift_chunk<T, W>(w[i], CXd(i), S);
      }
      collide_chunk<T, W>(w, par);
    }
    if (j >= 2 * (STEPS - 1)) {
      if (out && y0 + j - 2 * (STEPS - 1) < y1 &&
          bounds::ok(y0 >= 0 && y1 <= g.ny && x0 + (1 + fill) * V <= g.pitch,
                     bounds::ROWS_NODE)) {
#pragma unroll
        for (int i = 0; i < 9; ++i)
          *reinterpret_cast<Vec *>(drow + (long long)i * g.plane) = get_words(w[i]);
        for (int k = 1; k <= fill; ++k) {
#pragma unroll
          for (int i = 0; i < 9; ++i)
            *reinterpret_cast<Vec *>(drow + (long long)i * g.plane + k * V) = Vec{};
        }
      }
      drow += g.rstride;
    }
  }
}

// Register budgets, 64-thread blocks: 128 (116 used in FP32, 120 in 16 bits,
// no spills), 16 warps per SM, which their shared memory (13.8 KB per warp in
// FP32) allows too.  The FMA pipe is 70% busy on 8192^2 FP32 (251 GLUPS), with
// 54% of the issue slots used.  16 bits: chunks of eight nodes per lane took
// 210 registers, 8 warps, FMA pipe 65% (the conversions run on it); four nodes
// take the 128-lattice FP16 sweep from 43.3 to 42.1 ms.
template <typename T, int STEPS>
__global__ void __launch_bounds__(64, 8)
k_step_rows(const T *__restrict__ src, T *__restrict__ dst, Geom g, RowsGeom rg,
            typename PairParams<T>::type P, unsigned ntasks) {
  extern __shared__ uint4 rows_smem[];
  const unsigned warp = threadIdx.x >> 5, task = blockIdx.x * 2 + warp;
  pdl_wait();
  if (task >= ntasks) return;
  using Vec = typename RowsVec<T>::type;
  Vec *sm = reinterpret_cast<Vec *>(rows_smem) + warp * rows_smem_chunks(STEPS);
  if constexpr (sizeof(T) == 4)
    rows_task<T, STEPS>(src, dst, g, rg, P, task, threadIdx.x & 31, sm);
  else
    rows_task<T, STEPS>(src, dst, g, rg, ParamPairs{P}, task, threadIdx.x & 31, sm);
}

template <typename T, int STEPS>
cudaError_t launch_rows_steps(const Lattice &L, const void *src, void *dst, cudaStream_t st) {
  constexpr size_t smem = 2 * rows_smem_chunks(STEPS) * sizeof(typename RowsVec<T>::type);
  cudaError_t e = cudaFuncSetAttribute(
      k_step_rows<T, STEPS>, cudaFuncAttributeMaxDynamicSharedMemorySize, kMaxSmem);
  if (e != cudaSuccess) return e;
  const long long nt = L.rows.tasks;
  return launch_pdl(k_step_rows<T, STEPS>, (unsigned)((nt + 1) / 2), 64, smem, st,
                    static_cast<const T *>(src), static_cast<T *>(dst), L.g, L.rows,
                    pair_params<T>(L.dp), (unsigned)nt);
}

template <typename T>
cudaError_t launch_rows_t(const Lattice &L, const void *src, void *dst, cudaStream_t st,
                          int steps) {
  if (steps == 3) return launch_rows_steps<T, 3>(L, src, dst, st);
  if (steps == 2) return launch_rows_steps<T, 2>(L, src, dst, st);
  return cudaErrorInvalidValue;
}

// The batched form: every block reads its lattice's record and collision
// constants into shared memory (a lattice's constants cannot be kernel
// parameters here, and 25 broadcast pairs in registers would spill; read in
// pairs of 16 bytes: one by one the 128-lattice FP32 sweep took 52.9 instead
// of 49.3 ms), then its two warps take one task each.
template <typename T> struct RowsShared {
  RowsRec rec;
  alignas(16) float2 c[PC_COUNT];
  static constexpr int COUNT = PC_COUNT;
  static __device__ __forceinline__ float value(const DevParams &P, int k) {
    return pair_const(P, k);
  }
  __device__ __forceinline__ float2 *table() { return c; }
  __device__ __forceinline__ SharedPairs constants() const { return SharedPairs{c}; }
};

template <> struct RowsShared<float> {
  RowsRec rec;
  HlPairs pairs;
  static constexpr int COUNT = HL_COUNT;
  static __device__ __forceinline__ float value(const DevParams &P, int k) { return hl_const(P, k); }
  __device__ __forceinline__ float2 *table() { return pairs.c; }
  __device__ __forceinline__ const HlPairs &constants() const { return pairs; }
};

template <typename T>
__global__ void __maxnreg__(sizeof(T) == 4 ? 168 : 128)
k_rows_batch(const BatchEntry *__restrict__ ents, const RowsRec *__restrict__ recs, int nents,
             int parity, const int *__restrict__ limits, int k) {
  extern __shared__ uint4 rows_smem[];
  using Vec = typename RowsVec<T>::type;
  RowsShared<T> &S =
      *reinterpret_cast<RowsShared<T> *>(reinterpret_cast<Vec *>(rows_smem) +
                                         2 * rows_smem_chunks(kRowSteps));
  constexpr int NW = sizeof(RowsRec) / 4;
  static_assert(sizeof(RowsRec) % 4 == 0 && NW <= 64, "a record is copied one word per thread");
  if (threadIdx.x < NW)
    reinterpret_cast<uint32_t *>(&S.rec)[threadIdx.x] =
        reinterpret_cast<const uint32_t *>(recs + blockIdx.x)[threadIdx.x];
  pdl_wait();
  __syncthreads();
  const int lat = S.rec.lat;
  if (!bounds::ok(lat >= 0 && lat < nents, bounds::BATCH_REC)) return;
  if (limits != nullptr && k + kRowSteps > limits[lat]) return;  // block-uniform
  if (threadIdx.x < RowsShared<T>::COUNT) {
    const float v = RowsShared<T>::value(ents[lat].dp, threadIdx.x);
    S.table()[threadIdx.x] = make_float2(v, v);
  }
  __syncthreads();
  const RowsGeom &rg = S.rec.rg;
  const unsigned warp = threadIdx.x >> 5, task = S.rec.task + warp;
  if (task >= (unsigned)rg.tasks) return;
  const int from = parity ^ S.rec.off;
  rows_task<T, kRowSteps>(static_cast<const T *>(S.rec.buf[from]),
                          static_cast<T *>(S.rec.buf[from ^ 1]), S.rec.g, rg, S.constants(), task,
                          threadIdx.x & 31,
                          reinterpret_cast<Vec *>(rows_smem) + warp * rows_smem_chunks(kRowSteps));
}

template <typename T>
cudaError_t launch_rows_batch_t(const BatchList &bl, int parity, cudaStream_t st,
                                const int *limits, int k) {
  if (bl.nrows < 1) return cudaSuccess;
  constexpr size_t smem =
      2 * rows_smem_chunks(kRowSteps) * sizeof(typename RowsVec<T>::type) + sizeof(RowsShared<T>);
  cudaError_t e = cudaFuncSetAttribute(
      k_rows_batch<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, kMaxSmem);
  if (e != cudaSuccess) return e;
  return launch_pdl(k_rows_batch<T>, (unsigned)bl.nrows, 64, smem, st, bl.ents, bl.rows, bl.n,
                    parity, limits, k);
}

// ------------------------------------------------------------------ tile
// two adjacent nodes as stored
template <typename T> struct TilePair { using type = uint32_t; };
template <> struct TilePair<float> { using type = float2; };

// One stored node as raw bits, or an aligned pair, through L2 (the row may
// have been written by the launch before, see pdl_wait)
template <typename T>
__device__ __forceinline__ uint32_t node_bits(const T *p) {
  if constexpr (sizeof(T) == 4) return __ldcg(reinterpret_cast<const unsigned *>(p));
  else return __ldcg(reinterpret_cast<const unsigned short *>(p));
}
template <typename T>
__device__ __forceinline__ typename TilePair<T>::type node_pair(const T *a, const T *b) {
  if constexpr (sizeof(T) == 4)
    return make_float2(__uint_as_float(node_bits(a)), __uint_as_float(node_bits(b)));
  else
    return node_bits(a) | node_bits(b) << 16;
}

// nodes (j, j + 1), j even, of a row in shared memory, pulled from x - cx
template <typename T>
__device__ __forceinline__ F2 tile_pull(const T *row, int j, int cx) {
  if constexpr (sizeof(T) == 4) {
    if (cx == 0) {
      const float2 v = *reinterpret_cast<const float2 *>(row + j);
      return f2(v.x, v.y);
    }
    return cx == 1 ? f2(row[j - 1], row[j]) : f2(row[j + 1], row[j + 2]);
  } else {
    const uint32_t *w = reinterpret_cast<const uint32_t *>(row) + (j >> 1);
    uint32_t v;
    if (cx == 0) v = w[0];
    else if (cx == 1) v = __byte_perm(w[-1], w[0], 0x5432);
    else v = __byte_perm(w[0], w[1], 0x5432);
    float t[2];
    Elem<T>::unpack2(v, t);
    return f2(t[0], t[1]);
  }
}

template <typename T>
__device__ __forceinline__ void tile_store(T *p, F2 f) {
  float a, b;
  f2split(f, a, b);
  if constexpr (sizeof(T) == 4) *reinterpret_cast<float2 *>(p) = make_float2(a, b);
  else *reinterpret_cast<uint32_t *>(p) = Elem<T>::pack2(a, b);
}

// One tile: rows and columns of kTileCols nodes (32 lanes of two) with a
// halo of `steps` rows and `steps` columns (rounded up to even, so that a
// lane's pair is aligned in memory), both step buffers in shared memory, 9
// planes each.  Step s computes rows [s, H - s) of the tile, all 32 lanes;
// columns lose one valid node per side and step.  One warp takes a row, 16
// warps a block, one block an SM: the FMA pipe bounds it (16 rows of 64
// nodes take 800 of the 1200 - 1300 cycles measured per pass over them).
// A point source replaces the pulled populations of its node by `forced`
// (stored units, 9 per step).
template <typename T, bool FORCED>
__global__ void __launch_bounds__(kTileThreads, 1)
k_step_tile(const T *__restrict__ src, T *__restrict__ dst, Geom g, TileGeom tg,
            typename PairParams<T>::type P, int steps, const float *__restrict__ forced, int sx,
            int sy) {
  extern __shared__ __align__(16) unsigned char tile_smem[];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  constexpr int nw = kTileThreads / 32;
  const int ty = blockIdx.x / tg.ntx, tx = blockIdx.x - ty * tg.ntx;
  const int X0 = tx * tg.bx, Y0 = ty * tg.by;
  const int bw = min(tg.bx, g.nx - X0), bh = min(tg.by, g.ny - Y0);
  const int hx = tile_halo_x(steps), H = bh + 2 * steps;
  const int plane = H * kTileCols;
  // the shared memory is that of tg.by rows (block-uniform)
  if (!bounds::ok(bw >= 1 && bh >= 1 && bh <= tg.by && bw + 2 * hx <= kTileCols, bounds::TILE_NODE))
    return;
  T *A = reinterpret_cast<T *>(tile_smem), *B = A + 9 * plane;
  const int j = 2 * lane, x = X0 - hx + j;
  const bool need = j < bw + 2 * hx;
  auto wrap_y = [&](int y) {
    while (y < 0) y += g.ny;
    while (y >= g.ny) y -= g.ny;
    return bounds::ck(y, g.ny, bounds::TILE_NODE);
  };
  // the pair's nodes, each taken periodically, and which of them the source
  // is (-1: none)
  int xa = x;
  while (xa < 0) xa += g.nx;
  while (xa >= g.nx) xa -= g.nx;
  xa = bounds::ck(xa, g.nx, bounds::TILE_NODE);
  const int xb = xa + 1 == g.nx ? 0 : xa + 1;
  const bool vec = xa + 1 < g.nx && (xa & 1) == 0;
  const int at = FORCED ? (xa == sx ? 0 : (xb == sx ? 1 : -1)) : -1;
  pdl_wait();
  for (int r = warp; r < H; r += nw) {
    const T *row = src + (long long)wrap_y(Y0 - steps + r) * g.rstride;
    if (need) {
      using Pair = typename TilePair<T>::type;
      Pair v[9];
      if (vec) {
#pragma unroll
        for (int i = 0; i < 9; ++i)
          v[i] = __ldcg(reinterpret_cast<const Pair *>(row + (long long)i * g.plane + xa));
      } else {
#pragma unroll
        for (int i = 0; i < 9; ++i)
          v[i] = node_pair(row + (long long)i * g.plane + xa, row + (long long)i * g.plane + xb);
      }
#pragma unroll
      for (int i = 0; i < 9; ++i)
        *reinterpret_cast<Pair *>(A + i * plane + r * kTileCols + j) = v[i];
    }
  }
  __syncthreads();
  for (int s = 1; s <= steps; ++s) {
    for (int r = s + warp; r < H - s; r += nw) {
      F2 f[9];
#pragma unroll
      for (int i = 0; i < 9; ++i)
        f[i] = tile_pull<T>(A + i * plane + (r - CYd(i)) * kTileCols, j, CXd(i));
      if constexpr (FORCED) {
        if (at >= 0 && wrap_y(Y0 - steps + r) == sy) {
#pragma unroll
          for (int i = 0; i < 9; ++i) {
            const float v = forced[9 * (s - 1) + i];
            float a, b;
            f2split(f[i], a, b);
            f[i] = at == 0 ? f2(v, b) : f2(a, v);
          }
        }
      }
      if constexpr (sizeof(T) == 4) collide_two<T>(f, P);
      else collide_two<T>(f, ParamPairs{P});
      if (s < steps) {
#pragma unroll
        for (int i = 0; i < 9; ++i) tile_store<T>(B + i * plane + r * kTileCols + j, f[i]);
      } else if (j >= hx && j < hx + bw &&
                 bounds::ok(Y0 + r - steps >= 0 && Y0 + r - steps < g.ny && x >= 0 &&
                                x + 2 <= g.pitch,
                            bounds::TILE_NODE)) {
        // an odd row's last pair also writes its first padding column
        T *o = dst + (long long)(Y0 + r - steps) * g.rstride + x;
#pragma unroll
        for (int i = 0; i < 9; ++i) tile_store<T>(o + (long long)i * g.plane, f[i]);
      }
    }
    if (s < steps) {
      __syncthreads();
      T *t = A;
      A = B;
      B = t;
    }
  }
}

template <typename T, bool FORCED>
cudaError_t launch_tile_f(const Lattice &L, const void *src, void *dst, cudaStream_t st, int steps,
                          const float *forced, int sx, int sy) {
  const size_t smem = tile_bytes(L.tile.by, steps, (int)sizeof(T));
  cudaError_t e = cudaFuncSetAttribute(
      k_step_tile<T, FORCED>, cudaFuncAttributeMaxDynamicSharedMemorySize, kMaxSmem);
  if (e != cudaSuccess) return e;
  return launch_pdl(k_step_tile<T, FORCED>, (unsigned)(L.tile.ntx * L.tile.nty), kTileThreads,
                    smem, st, static_cast<const T *>(src), static_cast<T *>(dst), L.g, L.tile,
                    pair_params<T>(L.dp), steps, forced, sx, sy);
}

template <typename T>
cudaError_t launch_tile_t(const Lattice &L, const void *src, void *dst, cudaStream_t st, int steps,
                          const float *forced, int sx, int sy) {
  if (steps < 1 || steps > L.tile.steps) return cudaErrorInvalidValue;
  return forced ? launch_tile_f<T, true>(L, src, dst, st, steps, forced, sx, sy)
                : launch_tile_f<T, false>(L, src, dst, st, steps, nullptr, 0, 0);
}

}  // namespace lbm
