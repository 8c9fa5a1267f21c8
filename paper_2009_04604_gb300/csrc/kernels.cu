// kernels.cu -- instantiation and dispatch of the lattice Boltzmann kernels.
#include "step.cuh"

namespace lbm {

__global__ void k_reduce_final(const double *__restrict__ part, long long nblocks, int ncomp,
                               double *__restrict__ out) {
  // thread t sums partials t, t + 1024, ... of each component in order, then every warp
  // its lanes' sums and warp 0 the warps' (a tree of shuffles: the barrier tree over
  // 1024 sums took 13 us for three components, this takes 4)
  __shared__ double sm[32];
  const int t = threadIdx.x, lane = t & 31;
  chain_wait();
  for (int c = 0; c < ncomp; ++c) {
    double s = 0.0;
    for (long long b = t; b < nblocks; b += blockDim.x) s += part[b * ncomp + c];
    for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
    if (lane == 0) sm[t >> 5] = s;
    __syncthreads();
    if (t < 32) {
      s = lane < (int)(blockDim.x >> 5) ? sm[lane] : 0.0;
      for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
      if (lane == 0) out[c] = s;
    }
    __syncthreads();
  }
}

cudaError_t launch_reduce_final(const double *part, long long nblocks, int ncomp, double *out,
                                cudaStream_t s) {
  // no more warps than there are groups of 32 partials
  const int threads = (int)(nblocks >= 1024 ? 1024 : (nblocks + 31) / 32 * 32);
  return launch_chained(k_reduce_final, dim3(1), dim3(threads > 0 ? threads : 32), 0, s, true, part, nblocks, ncomp, out);
}

// Calls F.template operator()<L, S, M>() for the (lattice, dtype) pair.
template <class Fn>
static cudaError_t dispatch(int lattice, int dtype, Fn &&fn) {
  if (lattice == 0) {
    switch (dtype) {
      case 0: return fn.template operator()<D2Q9, double, double>();
      case 1: return fn.template operator()<D2Q9, float, float>();
      case 2: return fn.template operator()<D2Q9, __half, float>();
      case 3: return fn.template operator()<D2Q9, __nv_bfloat16, float>();
    }
  } else if (lattice == 1) {
    switch (dtype) {
      case 0: return fn.template operator()<D3Q19, double, double>();
      case 1: return fn.template operator()<D3Q19, float, float>();
      case 2: return fn.template operator()<D3Q19, __half, float>();
      case 3: return fn.template operator()<D3Q19, __nv_bfloat16, float>();
    }
  } else if (lattice == 2) {
    switch (dtype) {
      case 0: return fn.template operator()<D3Q27, double, double>();
      case 1: return fn.template operator()<D3Q27, float, float>();
      case 2: return fn.template operator()<D3Q27, __half, float>();
      case 3: return fn.template operator()<D3Q27, __nv_bfloat16, float>();
    }
  }
  return cudaErrorInvalidValue;
}

LBM_STEP_INSTANCES(LBM_STEP_DECLARE)

cudaError_t prepare_step_tma(int lattice, int dtype, int phys, int bx, int by, long long ntiles,
                             int *blocks, int *smem) {
  return dispatch(lattice, dtype, [&]<class L, typename S, typename M>() {
    return prepare_step_tma_ls<L, S>(phys, bx, by, ntiles, blocks, smem);
  });
}

cudaError_t launch_step(int lattice, int dtype, int variant, const View &v, const void *fin,
                        void *fout, const Launch &l, const Launch *lb) {
  return dispatch(lattice, dtype, [&]<class L, typename S, typename M>() {
    if (variant == 9 || variant == 10) return launch_split_ls<L, S>(variant, v, fin, fout, l, lb);
    if (variant >= 4 && variant <= 8) return launch_wide_ls<L, S>(variant, v, fin, fout, l);
    if (v.fused) return launch_bulk_ls<L, S>(variant, v, fin, fout, l, lb);
    return launch_one_ls<L, S>(variant, v, fin, fout, l);
  });
}

cudaError_t launch_step_batch(int lattice, int dtype, int variant, int kind, int phys, const BatchEntry *entries,
                              const int4 *tiles, int n, int T, int parity, const Launch &l) {
  return dispatch(lattice, dtype, [&]<class L, typename S, typename M>() {
    return launch_batch_ls<L, S>(variant, kind, phys, entries, tiles, n, T, parity, l);
  });
}

cudaError_t launch_init(int lattice, int dtype, const View &v, void *fout, double rho, double ux,
                        double uy, double uz, const Launch &l) {
  return dispatch(lattice, dtype, [&]<class L, typename S, typename M>() {
    k_init<L, S, M><<<l.grid, l.block, 0, l.stream>>>(v, static_cast<S *>(fout), rho, ux, uy, uz);
    return cudaGetLastError();
  });
}

cudaError_t launch_set_pop(int lattice, int dtype, const View &v, void *fout, const double *fh,
                           const Launch &l) {
  return dispatch(lattice, dtype, [&]<class L, typename S, typename M>() {
    k_set_pop<L, S, M><<<l.grid, l.block, 0, l.stream>>>(v, static_cast<S *>(fout), fh);
    return cudaGetLastError();
  });
}

cudaError_t launch_read(int lattice, int dtype, const View &v, const void *fin, double *fh,
                        double *rho, double *u, double *mass_part, const Launch &l) {
  return dispatch(lattice, dtype, [&]<class L, typename S, typename M>() {
    k_read<L, S, M><<<l.grid, l.block, 0, l.stream>>>(v, read_par(v), static_cast<const S *>(fin), fh, rho, u,
                                                      mass_part);
    return cudaGetLastError();
  });
}

// A body's records and a small lattice's: 8 to a warp, so that they spread over the SMs;
// else 32, whose links fill the lanes (128 x 96 x 80 duct, 43 thousand records: 11.3 us
// with 32, 16.5 with 8: the FP64 pipe takes an idle lane's time too). At most 4 blocks
// an SM: their partials are summed by one.
static constexpr long long kFewRecords = 5000;
int force_blocks(long long nrec) {
  const long long per_block = 8 * (nrec <= kFewRecords ? 8 : 32), n = (nrec + per_block - 1) / per_block;
  return (int)(n < 4 * kSMs ? n : 4 * kSMs);
}

cudaError_t launch_force(int lattice, int dtype, const View &v, const void *cur, const void *prev,
                         const RecSet &rs, long long nrec, const int *nrec_dev, int tag, double *part,
                         const Launch &l, double *tpart, double cx, double cy, double cz) {
  return dispatch(lattice, dtype, [&]<class L, typename S, typename M>() {
    auto *kern = nrec_dev != nullptr || nrec <= kFewRecords ? k_force<L, S, M, 8> : k_force<L, S, M, 32>;
    kern<<<l.grid, 256, 0, l.stream>>>(v, static_cast<const S *>(cur), static_cast<const S *>(prev), rs, nrec,
                                       nrec_dev, tag, part, tpart, cx, cy, cz);
    return cudaGetLastError();
  });
}

}  // namespace lbm
