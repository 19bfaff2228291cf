// lbm_batch3d.cuh - the 3-D step of a batch: the passes of the split step (lbm_kernels.cuh,
// lbm_n1.cuh), each one launch over the blocks of every instance.  A work list names the
// instance and the block of its own launch that a block stands for, the largest instances
// first; the instances' parameters and geometry are read from a table.
//
// Three launches of its own for every instance cost a launch's latency each.  us per step
// with those on four branches of the step's graph, with the persistent kernel before
// them, and in this form (FP32): 256 boxes of 8^3 1069, 140, 60; 256 of 16^3 1211, 454,
// 235; 64 of 32^3 602, 425, 316; 16 of 48^3 386, 534, 301; 4 of 64^3 163, 525, 160.  Boxes
// that fill the device by themselves pay for the parameters being read from memory: 4
// tubes of 64^3 220, 4266, 249.
#pragma once

#include "lbm_n1.cuh"

namespace lbm {

// One instance: what the passes of its step take as launch arguments in a single handle.
template <typename real> struct SplitInstance {
  Params p;
  void* pop[2];
  real *M, *W;
  NodeRange moments, nodes;                        // of the moments; of a collision by nodes or pairs
  int lo, hi, ncolx, ncoly, nseg;                  // columns and z-segments of the primitive fields
  int rowseg;                                      // segments of a row, of the collision by rows
  FastDiv drowseg, dny;
  unsigned units;                                  // shock capturing: units of the strain, columns of the coefficients
  FastDiv dunits;
  int n1tx, n1ty, n1seg;
  int ghosts;                                      // the collision leaves the ghost layers to the fill
};

// One block of a pass: an instance and the index of the block in the instance's own launch.
struct SplitItem {
  int inst;
  unsigned block;
};

template <typename S, typename real, bool RAGGED>
__global__ void __launch_bounds__(sizeof(real) == 8 ? 256 : 128)
k_moments_batch(const SplitInstance<real>* __restrict__ insts, const SplitItem* __restrict__ items, int parity) {
  wait_previous_launch();
  const SplitItem it = items[blockIdx.x];
  const SplitInstance<real>& in = insts[it.inst];
  const typename Store<S>::T* A = static_cast<const typename Store<S>::T*>(in.pop[parity]);
  if constexpr (sizeof(real) == 8) moments_nodes<3>(in.p, in.moments, A, in.M, it.block);
  else moments_groups<3, S, RAGGED>(in.p, in.moments, A, in.M, it.block);
}

template <typename real, class CL, int MINB>
__global__ void __launch_bounds__(kPrimX * kPrimY, MINB)
k_prims3_batch(const SplitInstance<real>* __restrict__ insts, const SplitItem* __restrict__ items) {
  wait_previous_launch();
  const SplitItem it = items[blockIdx.x];
  const SplitInstance<real>& in = insts[it.inst];
  prims_column<real, CL, MINB>(in.p, in.lo, in.hi, in.ncolx, in.ncoly, in.nseg, in.M, in.W, it.block);
}

template <typename S, bool BOUNDED, int W, int MINB>
__global__ void __launch_bounds__(W / 2, MINB)
k_collide_rows_batch(const SplitInstance<float>* __restrict__ insts, const SplitItem* __restrict__ items, int parity,
                     unsigned* errs) {
  wait_previous_launch();
  const SplitItem it = items[blockIdx.x];
  const SplitInstance<float>& in = insts[it.inst];
  collide_rows<3, S, kHandNothing, BOUNDED, W, MINB>(
      in.p, in.rowseg, in.drowseg, in.dny, static_cast<const typename Store<S>::T*>(in.pop[parity]),
      static_cast<typename Store<S>::T*>(in.pop[parity ^ 1]), in.M, in.W, errs + it.inst, it.block);
}

template <typename S, typename real, bool ODD, int NTB, int MINB>
__global__ void __launch_bounds__(NTB, MINB)
k_collide_batch(const SplitInstance<real>* __restrict__ insts, const SplitItem* __restrict__ items, int parity,
                unsigned* errs) {
  wait_previous_launch();
  const SplitItem it = items[blockIdx.x];
  const SplitInstance<real>& in = insts[it.inst];
  const typename Store<S>::T* A = static_cast<const typename Store<S>::T*>(in.pop[parity]);
  typename Store<S>::T* B = static_cast<typename Store<S>::T*>(in.pop[parity ^ 1]);
  if constexpr (sizeof(real) == 8)
    collide_nodes<3, S, real, kHandNothing, NTB, MINB>(in.p, in.nodes, A, B, in.M, in.W, errs + it.inst, it.block);
  else collide_pairs<3, S, kHandNothing, ODD, NTB, MINB>(in.p, in.nodes, A, B, in.M, in.W, errs + it.inst, it.block);
}

template <typename S, typename real>
__global__ void __launch_bounds__(128)
k_n1_strain_batch3(const SplitInstance<real>* __restrict__ insts, const SplitItem* __restrict__ items) {
  wait_previous_launch();
  const SplitItem it = items[blockIdx.x];
  const SplitInstance<real>& in = insts[it.inst];
  n1_strain_units<S, real>(in.p, in.units, in.dunits, in.dny, in.M, in.W, in.W + 3 * in.p.plane, it.block);
}

// the columns of the coefficients of a batch's instances (k_n1_coef_3d)
template <typename real> struct N1CoefBatch {
  const SplitInstance<real>* insts;
  const SplitItem* items;
  __device__ __forceinline__ N1CoefArgs<real> args() const {
    const SplitItem it = items[blockIdx.x];
    const SplitInstance<real>& in = insts[it.inst];
    return {in.p, in.M, in.W + 3 * in.p.plane, in.n1tx, in.n1ty, in.n1seg, it.block};
  }
};

// the ghost layers of the instances whose collision leaves them
template <typename S, typename real>
__global__ void k_ghosts_batch3(const SplitInstance<real>* __restrict__ insts, int parity) {
  wait_previous_launch();
  const SplitInstance<real>& in = insts[blockIdx.y];
  if (!in.ghosts) return;
  ghost_fill<3, S>(in.p, static_cast<typename Store<S>::T*>(in.pop[parity ^ 1]), blockIdx.x * (long long)blockDim.x + threadIdx.x,
                   (long long)gridDim.x * blockDim.x);
}

}  // namespace lbm
