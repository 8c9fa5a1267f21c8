// launch.hpp -- host-side entry points of the kernels (one per kernel family),
// dispatched on lattice and storage type.
#pragma once

#include <cuda_runtime.h>

#include "lattice.cuh"

namespace lbm {

constexpr int kSMs = 152;  // of a GB300: the launch rules count warps and blocks per SM

struct Launch {
  dim3 grid, block;
  cudaStream_t stream;
  int smem = 0;  // dynamic shared memory
};

// A kernel launch that, with chained, may begin while the kernel before it in the stream
// still runs (programmatic stream serialization): the kernel itself waits, by chain_wait,
// before it touches what that one reads or writes. Every kernel launched so calls
// chain_wait first. What it saves is the launch latency between short kernels.
template <class... P, class... A>
cudaError_t launch_chained(void (*kern)(P...), dim3 grid, dim3 block, int smem, cudaStream_t st, bool chained,
                           A &&...args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = (size_t)smem;
  cfg.stream = st;
  cudaLaunchAttribute at = {};
  at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at.val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = &at;
  cfg.numAttrs = chained ? 1 : 0;
  return cudaLaunchKernelEx(&cfg, kern, static_cast<P>(args)...);
}

// Sets the shared-memory limit of the TMA-staged step kernel for this launch shape
// and returns its persistent grid (SMs x resident blocks, at most ntiles) and its
// dynamic shared memory. Call outside stream capture.
// phys: PH_FORCE | PH_TRT bits of the view (see phys_of).
cudaError_t prepare_step_tma(int lattice, int dtype, int phys, int bx, int by, long long ntiles,
                             int *blocks, int *smem);

// lattice: 0 D2Q9, 1 D3Q19, 2 D3Q27; dtype: 0 F64, 1 F32, 2 F16, 3 BF16
// variant: the register budget and form of the step kernel (lbm_set_launch). 0..2: one
// node per thread at 80 registers, 3: 64, 11: 48, 12: 40, as the bulk step where v.fused,
// whose boundary kernel runs with the launch lb, else over the tile table; 4: the
// TMA-staged persistent kernel; 5, 6: two nodes per thread at 128 registers, 7: 80, 8: in
// 128-thread blocks at 72; 9 and 10: the split step, whose lattice kernel has 40 or 48
// and whose boundary kernel runs with the launch lb. FP64 has a single budget.
cudaError_t launch_step(int lattice, int dtype, int variant, const View &v, const void *fin,
                        void *fout, const Launch &l, const Launch *lb = nullptr);
// One launch of the batched step: n tiles of one kind and physics class (PH_FORCE |
// PH_TRT bits; boundary tiles have none), T consecutive ones per block; parity picks
// which buffer of each entry is read.
struct BatchEntry;
enum { kBatchBulk = 0, kBatchBoundary = 1, kBatchStep = 2 };
cudaError_t launch_step_batch(int lattice, int dtype, int variant, int kind, int phys, const BatchEntry *entries,
                              const int4 *tiles, int n, int T, int parity, const Launch &l);
cudaError_t launch_init(int lattice, int dtype, const View &v, void *fout, double rho, double ux,
                        double uy, double uz, const Launch &l);
cudaError_t launch_set_pop(int lattice, int dtype, const View &v, void *fout, const double *fh,
                           const Launch &l);
cudaError_t launch_read(int lattice, int dtype, const View &v, const void *fin, double *fh,
                        double *rho, double *u, double *mass_part, const Launch &l);
// Momentum-exchange partials over the records rs: nrec of them, or *nrec_dev
// (device) when nrec_dev is not null, in l.grid.x blocks (force_blocks(nrec), or any
// fixed number).
// cur is the state the last step wrote, prev the state it read (used for the
// links across thin shells; may be null when rs has none).
// With tpart, also the torque about (cx, cy, cz) of every link force, taken at the
// link's wall point x_F - q c_i (3 doubles per block).
int force_blocks(long long nrec);
cudaError_t launch_force(int lattice, int dtype, const View &v, const void *cur, const void *prev,
                         const RecSet &rs, long long nrec, const int *nrec_dev, int tag, double *part,
                         const Launch &l, double *tpart = nullptr, double cx = 0.0, double cy = 0.0,
                         double cz = 0.0);
// amask[n] of every padded node (View::amask) from the node kinds in v.flags
// (geometry.cu).
cudaError_t launch_amask(int lattice, const View &v, uint32_t *amask, cudaStream_t s);
cudaError_t launch_reduce_final(const double *part, long long nblocks, int ncomp, double *out,
                                cudaStream_t s);

}  // namespace lbm
