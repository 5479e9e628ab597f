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
//   k_step_rows  (large lattices, batches): each warp marches along y over a
//     strip of 30 chunks of V nodes, kRowSteps time levels deep; level l of
//     row y needs level l-1 of rows y-1, y, y+1, which the warp has just
//     computed, so intermediate levels live in lane-private shared-memory
//     slots and no warp waits for another.
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
  const float2 *c;
  __device__ __forceinline__ F2 operator()(PairConst k) const { return f2(c[k].x, c[k].y); }
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
// One lane's chunk of a plane (V nodes as four words) shifted by the x
// component of the plane's velocity: the missing element comes from the
// neighbouring lane, whose chunk is the neighbouring one.
template <typename T>
__device__ __forceinline__ void shift_chunk(uint32_t (&w)[4], int cx) {
  if (cx == 1) {
    const uint32_t prev = __shfl_up_sync(0xffffffffu, w[3], 1);
    if constexpr (sizeof(T) == 4) {
      w[3] = w[2]; w[2] = w[1]; w[1] = w[0]; w[0] = prev;
    } else {
      w[3] = __byte_perm(w[2], w[3], 0x5432);
      w[2] = __byte_perm(w[1], w[2], 0x5432);
      w[1] = __byte_perm(w[0], w[1], 0x5432);
      w[0] = __byte_perm(prev, w[0], 0x5432);
    }
  } else if (cx == -1) {
    const uint32_t next = __shfl_down_sync(0xffffffffu, w[0], 1);
    if constexpr (sizeof(T) == 4) {
      w[0] = w[1]; w[1] = w[2]; w[2] = w[3]; w[3] = next;
    } else {
      w[0] = __byte_perm(w[0], w[1], 0x5432);
      w[1] = __byte_perm(w[1], w[2], 0x5432);
      w[2] = __byte_perm(w[2], w[3], 0x5432);
      w[3] = __byte_perm(w[3], next, 0x5432);
    }
  }
}

// all nodes of a lane's chunk, two at a time
template <typename T, typename K>
__device__ __forceinline__ void collide_chunk(uint32_t (&w)[9][4], const K &P) {
  constexpr int PAIRS = sizeof(T) == 4 ? 2 : 4;
#pragma unroll
  for (int k = 0; k < PAIRS; ++k) {
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

__device__ __forceinline__ void set4(uint32_t (&w)[4], const uint4 &v) {
  w[0] = v.x; w[1] = v.y; w[2] = v.z; w[3] = v.w;
}
__device__ __forceinline__ uint4 get4(const uint32_t (&w)[4]) {
  return make_uint4(w[0], w[1], w[2], w[3]);
}

__device__ __forceinline__ void cp_async16(uint4 *smem, const void *g) {
  const unsigned a = (unsigned)__cvta_generic_to_shared(smem);
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(a), "l"(g) : "memory");
}

// Elements sh .. sh + V - 1 of chunk *a and the chunk `spare` slots after it
// (shared memory) laid end to end, the first `keep` of them replaced by w's.
template <typename T>
__device__ __forceinline__ void seam_chunk(uint32_t (&w)[4], const uint4 *a, int spare, int sh,
                                           int keep) {
  const uint32_t *p = reinterpret_cast<const uint32_t *>(a);
  constexpr int PER = 4 / (int)sizeof(T);  // elements per word
  const int k0 = sh / PER, far = 4 * spare - 4;
  uint32_t v[5];
#pragma unroll
  for (int q = 0; q < (PER == 2 ? 5 : 4); ++q) {
    const int k = k0 + q;  // at most 8: the funnel of an even shift ignores it
    v[q] = p[k < 4 ? k : min(k, 7) + far];
  }
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    if constexpr (PER == 2) {
      const uint32_t u = (sh & 1) ? __byte_perm(v[q], v[q + 1], 0x5432) : v[q];
      const uint32_t own = 2 * q + 1 < keep ? 0xffffffffu : (2 * q < keep ? 0xffffu : 0u);
      w[q] = (w[q] & own) | (u & ~own);
    } else {
      w[q] = q < keep ? w[q] : v[q];
    }
  }
}

// shared memory of one warp of k_step_rows, in 16-byte words: two stages of
// 9 incoming vectors and, per level boundary, 3 delayed by one row and 3 by
// two rows, for 32 lanes
constexpr int rows_smem_words(int steps) { return (18 + 9 * (steps - 1)) * 32; }

// Task `task` of a lattice (at least three chunks per row where V does not
// divide nx): strip task % strips of the chunks, rows
// [y0, y0 + rows).  Lane l holds the chunk of virtual nodes
// [(c0 - 1 + l) V, ... + V), taken periodically: lanes 1 .. cnt are the
// strip's own chunks, lanes 0 and cnt + 1 its halo.  After each level one
// more node of each halo chunk is invalid, so STEPS <= V levels leave the
// strip's nodes exact; in y each level loses one row per side, so level l
// (1 .. STEPS) covers rows y0 - (STEPS - l) .. y1 - 1 + (STEPS - l).
// In iteration j level 1 takes row y0 - (STEPS - 1) + j and level l the row
// l - 1 below it: its populations with c_y = -1 come from the row just
// computed (registers), those with c_y = 0 from the iteration before and
// those with c_y = +1 from two before (the delay slots, which only this
// lane touches: no synchronization).  Incoming rows are copied to shared
// memory one iteration ahead (cp.async), so no register holds a load in
// flight: with the loads in registers the compiler spilled (FP32 152 bytes
// at 168 registers) and the two-step form ran at 125 instead of 174 GLUPS.
// Where V does not divide the row length, up to three chunks of a row lie
// across its end (the halo chunk before node 0, the partial last chunk, the
// halo chunk after it): their lanes copy two aligned chunks, the second into
// the slot of an idle lane (strips are then at most 28 chunks wide), and
// assemble them.  A template on the seam, or element-wise gathers, ran
// ragged lattices at half the speed (4097 x 3071 FP16: 85 and 138 us per
// step).
template <typename T, int STEPS, typename K>
__device__ __forceinline__ void rows_task(const T *__restrict__ src, T *__restrict__ dst,
                                          const Geom &g, const RowsGeom &rg, const K &par,
                                          unsigned task, int lane, uint4 *sm) {
  constexpr int V = Elem<T>::V;
  static_assert(STEPS >= 2 && STEPS <= V, "the halo chunk covers V nodes");
  const unsigned seg = task / (unsigned)rg.strips, strip = task - seg * (unsigned)rg.strips;
  const int y0 = (int)seg * rg.rows, y1 = min(y0 + rg.rows, g.ny);
  const int c0 = (int)strip * rg.width, cnt = min(rg.width, g.nchunks - c0);
  const bool in = lane < cnt + 2, out = lane >= 1 && lane <= cnt;
  const int vc = in ? c0 - 1 + lane : 0, vx = vc * V;  // chunk, first virtual node
  const int part = g.nx & (V - 1);  // nodes of a partial last chunk (0: none)
  int ca = vc < 0 ? vc + g.nchunks : (vc >= g.nchunks ? vc - g.nchunks : vc), cb = 0;
  // seam lanes: element e of the chunk is element e + sh of the chunks ca, cb
  // laid end to end (a partial last chunk keeps its own first `part`)
  const bool seam = in && part != 0 && (vc < 0 || vc >= g.nchunks - 1);
  int sh = 0, spare = 0;
  if (seam) {
    sh = vc < 0 ? part : V - part;
    if (vc < 0) ca = g.nchunks - 2;
    cb = vc < 0 ? g.nchunks - 1 : (vc == g.nchunks ? 1 : 0);
    // (vc < 0 and vc = nchunks share a warp only in a lattice of one strip)
    spare = 31 - (vc < 0 ? 0 : (vc == g.nchunks - 1 ? 1 : (rg.strips == 1 ? 2 : 0))) - lane;
  }
  const int x0 = ca * V;
  const int ya = y0 - (STEPS - 1);
  const int n = y1 - y0 + 2 * (STEPS - 1);
  auto row_of = [&](int y) -> const T * {
    while (y < 0) y += g.ny;
    while (y >= g.ny) y -= g.ny;
    return src + (long long)y * g.rstride;
  };
  uint4 *raw = sm + lane, *dly = sm + 18 * 32 + lane;
  const T *pm = row_of(ya - 1) + x0, *pc = row_of(ya) + x0, *pp = row_of(ya + 1) + x0;
  int fetched = 0;
  auto fetch = [&]() {  // level 1's row ya + fetched into stage fetched & 1
    if (fetched < n) {
      uint4 *q = raw + (fetched & 1) * (9 * 32);
      if (in) {  // an idle lane's slots may be a seam lane's
#pragma unroll
        for (int i = 0; i < 9; ++i) {
          const T *row = (CYd(i) == 1 ? pm : (CYd(i) == -1 ? pp : pc)) + (long long)i * g.plane;
          cp_async16(q + i * 32, row);
        }
      }
      if (seam) {
#pragma unroll
        for (int i = 0; i < 9; ++i) {
          const T *row = (CYd(i) == 1 ? pm : (CYd(i) == -1 ? pp : pc)) + (long long)i * g.plane;
          cp_async16(q + i * 32 + spare, row + (cb - ca) * V);
        }
      }
      ++fetched;
      pm = pc;
      pc = pp;
      pp = row_of(ya + 1 + fetched) + x0;
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  fetch();
  T *drow = dst + (long long)y0 * g.rstride + (out ? vx : 0);
  const bool fill = (g.nchunks & 1) && out && vx + V >= g.nx;  // see fills_sector
  for (int j = 0; j < n; ++j) {
    fetch();
    asm volatile("cp.async.wait_group 1;" ::: "memory");
    uint32_t w[9][4];
    {
      const uint4 *q = raw + (j & 1) * (9 * 32);
#pragma unroll
      for (int i = 0; i < 9; ++i) set4(w[i], q[i * 32]);
      if (seam) {
#pragma unroll
        for (int i = 0; i < 9; ++i)
          seam_chunk<T>(w[i], q + i * 32, spare, sh, vc == g.nchunks - 1 ? part : 0);
      }
    }
#pragma unroll
    for (int i = 0; i < 9; ++i) shift_chunk<T>(w[i], CXd(i));
    collide_chunk<T>(w, par);
#pragma unroll
    for (int l = 1; l < STEPS; ++l) {
      if (j < 2 * (l - 1)) break;  // level l has no row yet
      uint4 *a = dly + (l - 1) * (9 * 32), *b = a + (3 + 3 * (j & 1)) * 32;
      uint32_t u[9][4];
      set4(u[0], a[0]); set4(u[1], a[32]); set4(u[3], a[64]);
      set4(u[2], b[0]); set4(u[5], b[32]); set4(u[6], b[64]);
      a[0] = get4(w[0]); a[32] = get4(w[1]); a[64] = get4(w[3]);
      b[0] = get4(w[2]); b[32] = get4(w[5]); b[64] = get4(w[6]);
      if (j < 2 * l) break;
#pragma unroll
      for (int i = 0; i < 9; ++i) {
        if (CYd(i) != -1) {
#pragma unroll
          for (int q = 0; q < 4; ++q) w[i][q] = u[i][q];
        }
        shift_chunk<T>(w[i], CXd(i));
      }
      collide_chunk<T>(w, par);
    }
    if (j >= 2 * (STEPS - 1)) {
      if (out) {
#pragma unroll
        for (int i = 0; i < 9; ++i)
          *reinterpret_cast<uint4 *>(drow + (long long)i * g.plane) = get4(w[i]);
        if (fill) {
#pragma unroll
          for (int i = 0; i < 9; ++i)
            *reinterpret_cast<uint4 *>(drow + (long long)i * g.plane + V) = make_uint4(0, 0, 0, 0);
        }
      }
      drow += g.rstride;
    }
  }
}

// Register budgets: 64-thread blocks, 168 registers (FP32; no spills, 12
// warps per SM) or 255 (16 bits: 224, 8 warps; at 168 it spills 24 bytes).
template <typename T, int STEPS>
__global__ void __launch_bounds__(64, sizeof(T) == 4 ? 6 : 4)
k_step_rows(const T *__restrict__ src, T *__restrict__ dst, Geom g, RowsGeom rg,
            typename PairParams<T>::type P, unsigned ntasks) {
  extern __shared__ uint4 rows_smem[];
  const unsigned warp = threadIdx.x >> 5, task = blockIdx.x * 2 + warp;
  pdl_wait();
  if (task >= ntasks) return;
  uint4 *sm = rows_smem + warp * rows_smem_words(STEPS);
  if constexpr (sizeof(T) == 4)
    rows_task<T, STEPS>(src, dst, g, rg, P, task, threadIdx.x & 31, sm);
  else
    rows_task<T, STEPS>(src, dst, g, rg, ParamPairs{P}, task, threadIdx.x & 31, sm);
}

template <typename T, int STEPS>
cudaError_t launch_rows_steps(const Lattice &L, const void *src, void *dst, cudaStream_t st) {
  constexpr size_t smem = 2 * rows_smem_words(STEPS) * sizeof(uint4);
  cudaError_t e = cudaFuncSetAttribute(
      k_step_rows<T, STEPS>, cudaFuncAttributeMaxDynamicSharedMemorySize, kMaxSmem);
  if (e != cudaSuccess) return e;
  const long long nt = (long long)L.rows.strips * ((L.g.ny + L.rows.rows - 1) / L.rows.rows);
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
  T *A = reinterpret_cast<T *>(tile_smem), *B = A + 9 * plane;
  const int j = 2 * lane, x = X0 - hx + j;
  const bool need = j < bw + 2 * hx;
  auto wrap_y = [&](int y) {
    while (y < 0) y += g.ny;
    while (y >= g.ny) y -= g.ny;
    return y;
  };
  // the pair's nodes, each taken periodically, and which of them the source
  // is (-1: none)
  int xa = x;
  while (xa < 0) xa += g.nx;
  while (xa >= g.nx) xa -= g.nx;
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
      } else if (j >= hx && j < hx + bw) {
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
