// step.cuh -- launch of the fused step kernel for one (lattice, storage type).
//
// The step kernel has many instantiations (register budget, node pairs, force
// path, the TMA-staged kernel). They are compiled in three translation units per
// (lattice, storage type), step_inst.cu built once for each part of each pair, so
// that the build runs them in parallel: the one-node kernels (launch_one_ls), the
// node pairs and the TMA-staged kernel (launch_wide_ls), and the bulk step with
// the split and the batched step (launch_bulk_ls, launch_split_ls, launch_batch_ls). kernels.cu
// dispatches to them.
#pragma once

#include "kernels.cuh"
#include "launch.hpp"

namespace lbm {

// Compile-time physics (PH_FORCE, PH_TRT) of a view.
inline int phys_of(const View &v) { return (v.has_force ? PH_FORCE : 0) | (v.trt ? PH_TRT : 0); }

// The step grid is 1-D, one block per entry of the tile table (l.grid.x entries).
template <class L, typename S, typename M, int MINB, bool PAIR = false, int MAXT = 256>
cudaError_t step_variant(const View &v, const void *fin, void *fout, const Launch &l) {
  const S *a = static_cast<const S *>(fin);
  S *b = static_cast<S *>(fout);
  switch (phys_of(v)) {
    case PH_FORCE: k_step<L, S, M, MINB, PH_FORCE, PAIR, MAXT><<<l.grid, l.block, l.smem, l.stream>>>(v, a, b); break;
    case PH_TRT: k_step<L, S, M, MINB, PH_TRT, PAIR, MAXT><<<l.grid, l.block, l.smem, l.stream>>>(v, a, b); break;
    case PH_FORCE | PH_TRT:
      k_step<L, S, M, MINB, PH_FORCE | PH_TRT, PAIR, MAXT><<<l.grid, l.block, l.smem, l.stream>>>(v, a, b);
      break;
    default: k_step<L, S, M, MINB, 0, PAIR, MAXT><<<l.grid, l.block, l.smem, l.stream>>>(v, a, b); break;
  }
  return cudaGetLastError();
}

// The boundary kernel of the split and the bulk step, on lb->stream (where lb is given).
// The caller orders the two streams around the pair of kernels.
template <class L, typename S, typename M>
cudaError_t boundary_launch(const View &v, const void *fin, void *fout, const Launch *lb) {
  if (lb == nullptr || lb->grid.x == 0) return cudaSuccess;
  k_boundary<L, S, M><<<lb->grid, lb->block, lb->smem, lb->stream>>>(v, static_cast<const S *>(fin),
                                                                     static_cast<S *>(fout));
  return cudaGetLastError();
}

// The split step (variants 9, 10): the boundary kernel, then the lattice kernel on l.stream.
template <class L, typename S, typename M, int MINB>
cudaError_t split_variant(const View &v, const void *fin, void *fout, const Launch &l, const Launch *lb) {
  const S *a = static_cast<const S *>(fin);
  S *b = static_cast<S *>(fout);
  cudaError_t e = boundary_launch<L, S, M>(v, fin, fout, lb);
  if (e != cudaSuccess) return e;
  switch (phys_of(v)) {
    case PH_FORCE: k_lattice<L, S, M, MINB, PH_FORCE><<<l.grid, l.block, 0, l.stream>>>(v, a, b); break;
    case PH_TRT: k_lattice<L, S, M, MINB, PH_TRT><<<l.grid, l.block, 0, l.stream>>>(v, a, b); break;
    case PH_FORCE | PH_TRT: k_lattice<L, S, M, MINB, PH_FORCE | PH_TRT><<<l.grid, l.block, 0, l.stream>>>(v, a, b); break;
    default: k_lattice<L, S, M, MINB, 0><<<l.grid, l.block, 0, l.stream>>>(v, a, b); break;
  }
  return cudaGetLastError();
}

// The bulk step: the boundary kernel for what is left to it, then the bulk kernel, whose
// grid is the lattice (l.grid: x tiles, groups of y tiles, planes).
template <class L, typename S, typename M, int MINB>
cudaError_t bulk_variant(const View &v, const void *fin, void *fout, const Launch &l, const Launch *lb) {
  cudaError_t e = boundary_launch<L, S, M>(v, fin, fout, lb);
  if (e != cudaSuccess) return e;
  Planes p;
  for (int i = 0; i < L::Q; ++i) {  // an integer sum: a shifted plane may begin before its buffer
    p.src[i] = reinterpret_cast<const void *>(reinterpret_cast<uintptr_t>(fin) + (long long)v.loff[i] * (long long)sizeof(S));
    p.dst[i] = static_cast<S *>(fout) + v.soff[i];
  }
  p.fin = fin;
  p.fout = fout;
  switch (phys_of(v)) {
    case PH_FORCE: k_bulk<L, S, M, MINB, PH_FORCE><<<l.grid, l.block, l.smem, l.stream>>>(v, p); break;
    case PH_TRT: k_bulk<L, S, M, MINB, PH_TRT><<<l.grid, l.block, l.smem, l.stream>>>(v, p); break;
    case PH_FORCE | PH_TRT: k_bulk<L, S, M, MINB, PH_FORCE | PH_TRT><<<l.grid, l.block, l.smem, l.stream>>>(v, p); break;
    default: k_bulk<L, S, M, MINB, 0><<<l.grid, l.block, l.smem, l.stream>>>(v, p); break;
  }
  return cudaGetLastError();
}

// Shared-memory bytes of one stage of the TMA-staged step: the rows of every
// population plane with a 16-byte halo on each side, the flag rows, and at least
// the boundary tiles' staging array.
template <class L, typename S, typename M>
int tma_stage_bytes(int bx, int by) {
  const int halo = 16 / (int)sizeof(S);
  const int pops = L::Q * by * (bx + 2 * halo) * (int)sizeof(S);
  const int need = pops + bx * by;
  const int stagebnd = L::Q * 256 * (int)sizeof(M);
  const int b = need > stagebnd ? need : stagebnd;
  return (b + 127) / 128 * 128;
}

// Two persistent blocks per SM, each with as many stages as half of the shared
// memory allows (at most 16): the copies in flight, not registers, then set the
// memory-level parallelism.
inline int tma_stages(int stage_bytes, int optin) {
  int k = (optin / 2 - 128) / stage_bytes;
  return k > 16 ? 16 : k;
}

template <class L, typename S, typename M, int PHYS>
cudaError_t tma_prepare(int bx, int by, long long ntiles, int *blocks, int *smem) {
  const int sb = tma_stage_bytes<L, S, M>(bx, by);
  int dev0 = 0, optin = 0;
  cudaError_t e0 = cudaGetDevice(&dev0);
  if (e0 == cudaSuccess) e0 = cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev0);
  if (e0 != cudaSuccess) return e0;
  const int stages = tma_stages(sb, optin);
  if (stages < 2) return cudaErrorInvalidConfiguration;
  *smem = 128 + stages * sb;
  auto kern = k_step_tma<L, S, M, PHYS>;
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, *smem);
  if (e != cudaSuccess) return e;
  int dev = 0, nsm = 0, per = 0;
  e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
  if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, kern, bx * by, *smem);
  if (e != cudaSuccess) return e;
  if (per < 1) return cudaErrorInvalidConfiguration;
  long long b = (long long)nsm * per;
  if (b > ntiles) b = ntiles;
  *blocks = (int)(b < 1 ? 1 : b);
  return cudaSuccess;
}

template <class L, typename S, typename M, int PHYS>
cudaError_t tma_launch(const View &v, const void *fin, void *fout, const Launch &l) {
  const int sb = tma_stage_bytes<L, S, M>(l.block.x, l.block.y);
  const int stages = (l.smem - 128) / sb;
  k_step_tma<L, S, M, PHYS><<<l.grid, l.block, l.smem, l.stream>>>(
      v, static_cast<const S *>(fin), static_cast<S *>(fout), stages, sb);
  return cudaGetLastError();
}

// Storage type S of lattice L: M is the arithmetic type (FP64 for FP64 storage).
template <typename S> struct MathOf { using T = float; };
template <> struct MathOf<double> { using T = double; };

// Register budgets: variants 0..2 share one kernel. At 80 registers (3 resident
// 256-thread blocks) no one-node kernel of any lattice spills, so the looser
// budgets of variants 0 and 1 would only lower the number of resident warps.
// Variants 5 and 6 share one in the same way (two blocks, 128 registers).
template <class L, typename S>
cudaError_t launch_one_ls(int variant, const View &v, const void *fin, void *fout, const Launch &l) {
  using M = typename MathOf<S>::T;
  if constexpr (sizeof(M) == 8) {
    return step_variant<L, S, M, 1>(v, fin, fout, l);  // FP64: one register budget
  } else {
    switch (variant) {
      case 3: return step_variant<L, S, M, 4>(v, fin, fout, l);
      case 11: return step_variant<L, S, M, 5>(v, fin, fout, l);
      case 12: return step_variant<L, S, M, 6>(v, fin, fout, l);
      default: return step_variant<L, S, M, 3>(v, fin, fout, l);
    }
  }
}

// The same variants as the bulk step (View::fused).
template <class L, typename S>
cudaError_t launch_bulk_ls(int variant, const View &v, const void *fin, void *fout, const Launch &l,
                            const Launch *lb) {
  using M = typename MathOf<S>::T;
  if constexpr (sizeof(M) == 8) {
    return bulk_variant<L, S, M, 1>(v, fin, fout, l, lb);
  } else {
    switch (variant) {
      case 3: return bulk_variant<L, S, M, 4>(v, fin, fout, l, lb);
      case 11: return bulk_variant<L, S, M, 5>(v, fin, fout, l, lb);
      case 12: return bulk_variant<L, S, M, 6>(v, fin, fout, l, lb);
      default: return bulk_variant<L, S, M, 3>(v, fin, fout, l, lb);
    }
  }
}

template <class L, typename S>
cudaError_t launch_wide_ls(int variant, const View &v, const void *fin, void *fout, const Launch &l) {
  using M = typename MathOf<S>::T;
  if constexpr (sizeof(M) == 8) {
    return cudaErrorInvalidValue;
  } else {
    if (variant == 4) {
      switch (phys_of(v)) {
        case PH_FORCE: return tma_launch<L, S, M, PH_FORCE>(v, fin, fout, l);
        case PH_TRT: return tma_launch<L, S, M, PH_TRT>(v, fin, fout, l);
        case PH_FORCE | PH_TRT: return tma_launch<L, S, M, PH_FORCE | PH_TRT>(v, fin, fout, l);
        default: return tma_launch<L, S, M, 0>(v, fin, fout, l);
      }
    }
    if (variant == 7) return step_variant<L, S, M, 3, true>(v, fin, fout, l);
    if (variant == 8) return step_variant<L, S, M, 7, true, 128>(v, fin, fout, l);
    return step_variant<L, S, M, 2, true>(v, fin, fout, l);
  }
}

template <class L, typename S>
cudaError_t launch_split_ls(int variant, const View &v, const void *fin, void *fout, const Launch &l,
                            const Launch *lb) {
  using M = typename MathOf<S>::T;
  if constexpr (sizeof(M) == 8) return cudaErrorInvalidValue;
  else if (variant == 9) return split_variant<L, S, M, 6>(v, fin, fout, l, lb);
  else return split_variant<L, S, M, 5>(v, fin, fout, l, lb);
}

// Kernels of the batched step for one physics class. FP64 on D3Q19 in blocks of 256
// threads stages just 48 KB, which with a kernel's static copy of an entry passes the
// default limit of 48 KB.
template <class Kern>
cudaError_t batch_kernel(Kern kern, const BatchEntry *e, const int4 *tiles, int n, int T, int parity,
                         const Launch &l) {
  if (l.smem + (int)(sizeof(BatchEntry)) > 48 * 1024) {
    const cudaError_t r = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, l.smem);
    if (r != cudaSuccess) return r;
  }
  kern<<<l.grid, l.block, l.smem, l.stream>>>(e, tiles, n, T, parity);
  return cudaGetLastError();
}

template <class L, typename S, typename M, int MINB, bool BULK, int PHYS>
cudaError_t batch_phys(const BatchEntry *e, const int4 *tiles, int n, int T, int parity, const Launch &l) {
  if constexpr (BULK) return batch_kernel(k_bulk_batch<L, S, M, MINB, PHYS>, e, tiles, n, T, parity, l);
  else return batch_kernel(k_step_batch<L, S, M, MINB, PHYS>, e, tiles, n, T, parity, l);
}

template <class L, typename S, typename M, int MINB, bool BULK>
cudaError_t batch_variant(int phys, const BatchEntry *e, const int4 *tiles, int n, int T, int parity,
                          const Launch &l) {
  switch (phys) {
    case PH_FORCE: return batch_phys<L, S, M, MINB, BULK, PH_FORCE>(e, tiles, n, T, parity, l);
    case PH_TRT: return batch_phys<L, S, M, MINB, BULK, PH_TRT>(e, tiles, n, T, parity, l);
    case PH_FORCE | PH_TRT: return batch_phys<L, S, M, MINB, BULK, PH_FORCE | PH_TRT>(e, tiles, n, T, parity, l);
    default: return batch_phys<L, S, M, MINB, BULK, 0>(e, tiles, n, T, parity, l);
  }
}

// kind: the tiles of the fused simulations (kBatchBulk), their boundary tiles
// (kBatchBoundary, one per block), or the other simulations' tiles (kBatchStep).
// Register budgets: bulk tiles 64, and 48 for variant 3; the other simulations' tiles
// 80, and 64 for variant 3.
template <class L, typename S>
cudaError_t launch_batch_ls(int variant, int kind, int phys, const BatchEntry *e, const int4 *tiles, int n, int T,
                            int parity, const Launch &l) {
  using M = typename MathOf<S>::T;
  if (kind == kBatchBoundary) {
    k_boundary_batch<L, S, M><<<l.grid, l.block, l.smem, l.stream>>>(e, tiles, parity);
    return cudaGetLastError();
  }
  if constexpr (sizeof(M) == 8) {
    if (kind == kBatchBulk) return batch_variant<L, S, M, 1, true>(phys, e, tiles, n, T, parity, l);
    return batch_variant<L, S, M, 1, false>(phys, e, tiles, n, T, parity, l);
  } else {
    if (kind == kBatchBulk) {
      if (variant == 3) return batch_variant<L, S, M, 5, true>(phys, e, tiles, n, T, parity, l);
      return batch_variant<L, S, M, 4, true>(phys, e, tiles, n, T, parity, l);
    }
    if (variant == 3) return batch_variant<L, S, M, 4, false>(phys, e, tiles, n, T, parity, l);
    return batch_variant<L, S, M, 3, false>(phys, e, tiles, n, T, parity, l);
  }
}

template <class L, typename S>
cudaError_t prepare_step_tma_ls(int phys, int bx, int by, long long ntiles, int *blocks, int *smem) {
  using M = typename MathOf<S>::T;
  if constexpr (sizeof(M) == 8) {
    return cudaErrorInvalidValue;  // FP64 has no TMA-staged variant
  } else {
    switch (phys) {
      case PH_FORCE: return tma_prepare<L, S, M, PH_FORCE>(bx, by, ntiles, blocks, smem);
      case PH_TRT: return tma_prepare<L, S, M, PH_TRT>(bx, by, ntiles, blocks, smem);
      case PH_FORCE | PH_TRT: return tma_prepare<L, S, M, PH_FORCE | PH_TRT>(bx, by, ntiles, blocks, smem);
      default: return tma_prepare<L, S, M, 0>(bx, by, ntiles, blocks, smem);
    }
  }
}

#define LBM_STEP_INSTANCES(X) \
  X(D2Q9, double) X(D2Q9, float) X(D2Q9, __half) X(D2Q9, __nv_bfloat16) \
  X(D3Q19, double) X(D3Q19, float) X(D3Q19, __half) X(D3Q19, __nv_bfloat16) \
  X(D3Q27, double) X(D3Q27, float) X(D3Q27, __half) X(D3Q27, __nv_bfloat16)

#define LBM_STEP_PART0(X, Lat, Sto) \
  X template cudaError_t launch_one_ls<Lat, Sto>(int, const View &, const void *, void *, const Launch &);
#define LBM_STEP_PART1(X, Lat, Sto)                                                                       \
  X template cudaError_t launch_wide_ls<Lat, Sto>(int, const View &, const void *, void *, const Launch &); \
  X template cudaError_t prepare_step_tma_ls<Lat, Sto>(int, int, int, long long, int *, int *);
#define LBM_STEP_PART2(X, Lat, Sto)                                                              \
  X template cudaError_t launch_bulk_ls<Lat, Sto>(int, const View &, const void *, void *, const Launch &, \
                                                   const Launch *);                              \
  X template cudaError_t launch_split_ls<Lat, Sto>(int, const View &, const void *, void *, const Launch &, \
                                                   const Launch *);                              \
  X template cudaError_t launch_batch_ls<Lat, Sto>(int, int, int, const BatchEntry *, const int4 *, int, int, int, \
                                                   const Launch &);
#define LBM_STEP_DECLARE(Lat, Sto)      \
  LBM_STEP_PART0(extern, Lat, Sto)      \
  LBM_STEP_PART1(extern, Lat, Sto)      \
  LBM_STEP_PART2(extern, Lat, Sto)

}  // namespace lbm
