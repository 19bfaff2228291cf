// lbm_internal.cuh - handle, kernel parameters and the dispatch table that
// the C interface (lbm_capi.cu) uses to reach the per-lattice /
// per-precision kernel instantiations (k_*.cu).
#pragma once

#include <cuda_runtime.h>
#include <cuda_fp16.h>
#include <stdint.h>
#include <stddef.h>

#include "../../include/lbm.h"
#include "lbm_device.cuh"

namespace lbm {

constexpr int kGhost = 4;         // ghost layers per non-periodic x face
constexpr int kMaxPartials = 1024;
constexpr unsigned kFlagWait = LBM_FLAG_INCOMPLETE;   // a bounded wait for an asynchronous copy ran out
constexpr int kMaxTiles = 16;     // tile candidates whose autotune times are kept

// Everything a kernel needs, passed by value.
struct Params {
  // geometry: padded x index xp = x + G; node offset = (z*Ny + y)*pitch + xp
  int D, Q, Nx, Ny, Nz, G, pitch;
  long long plane;            // elements per population plane = Nz*Ny*pitch
  int periodic_x;
  int bc_lo, bc_hi;           // LBM_BC_* of the x faces
  // model (FP64 master copy)
  double a, b, R, cv, kappa, eta_over_mu, mu, k_over_mu;
  int eos_kind;               // LBM_EOS_VDW | LBM_EOS_PR
  double Tc, mpr;             // Peng-Robinson T_c and alpha slope
  // inflow states (rho, u[3], T) and their equilibria (post-collision ghosts);
  // wall faces: (unused, u[3], T) of the wall
  double st_lo[5], st_hi[5];
  double eq_lo[54], eq_hi[54];   // f then g
  // FP16-deviation reference populations (f then g)
  float ref[54];
  float refsum[2];               // their sums over f and over g
  // learned closure: device inference image (mlp::Image), NULL for the exact closure
  const void* mlp;
  // shock capturing (Sec. 4.4): on/off, coefficients C_mu, C_eta, C_k; the step
  // reads the numerical mu, eta, k of the node from sc_visc (3 planes, work planes
  // after them); the 2-D step writes rho and T (batches: u too) to sc_prims (4
  // planes), all in compute precision on the padded plane layout
  int sc_on;
  double sc_c[3];
  void* sc_prims;
  const void* sc_visc;
  // FP64 temperature inversion in FP32 arithmetic (lbm_set_temperature_fp64);
  // read by AnyClosure (the steps select their closure instead)
  int t64;
  // the handle's two population buffers (2 Q plane elements each): the
  // bounds of every population access in bounds-check builds
  const void* pop[2];
#ifdef LBM_BOUNDS_CHECK
  // elements [hide_lo, hide_hi) of both buffers that count as outside (for tests)
  long long hide_lo, hide_hi;
#endif
  // the model constants above rounded to FP32 once on the host (set_model_fp32),
  // so that FP32 kernels read them as they are instead of converting the FP64
  // copies (a conversion the compiler may repeat inside loops, on the FP64 pipe)
  Model<float> mf;
};

template <typename real> __host__ __device__ inline Model<real> model_convert(const Params& p) {
  Model<real> m;
  m.a = real(p.a); m.b = real(p.b); m.R = real(p.R); m.cv = real(p.cv);
  m.kappa = real(p.kappa); m.eta_over_mu = real(p.eta_over_mu);
  m.mu = real(p.mu); m.k_over_mu = real(p.k_over_mu);
  m.kind = p.eos_kind; m.Tc = real(p.Tc); m.mpr = real(p.mpr);
  return m;
}

// model constants in the arithmetic type
template <typename real> __host__ __device__ inline Model<real> model_of(const Params& p) {
  if constexpr (sizeof(real) == 4) return p.mf;
  else return model_convert<real>(p);
}

// fill Params::mf from the FP64 constants (after every change of them)
inline void set_model_fp32(Params& p) { p.mf = model_convert<float>(p); }

constexpr int kIncomplete = 2;

// One solver instance.
struct Handle {
  int D, Q, Nx, Ny, Nz;
  lbm_eos eos;
  double tau, Pr, cv;
  Params p;
  int precision;
  size_t elem_bytes;          // bytes per stored population value
  void* pop[2];               // ping-pong population buffers
  int cur;                    // index of the buffer holding the current state
  void* scratch;              // moment / primitive fields of the split step and the reported fields
  size_t scratch_bytes;
  double* partials;           // kMaxPartials*(D+2) reduction partials
  double* totals_dev;         // D+2
  unsigned* err_dev;          // sticky status word
  unsigned* err_host;         // pinned
  double* io_dev;             // staging for host <-> device field copies
  size_t io_bytes;
  cudaStream_t stream;
  int initialized, unstable;  // unstable: 1 a fatal flag, kIncomplete the state is lost
  int unchecked;              // steps enqueued since the status word was last read
  int step_kernel;            // LBM_STEP_FUSED | LBM_STEP_MULTIPASS
  int tile_cfg;               // index of the step's candidate (lbm_autotune)
  long long launches;
  int closure;                // LBM_CLOSURE_EXACT | LBM_CLOSURE_MLP
  void* mlp_img;              // device copy of the attached network's inference image
  float tune_ms[kMaxTiles];    // ms per step of every candidate at the last lbm_autotune
  int tune_n;
  int use_graphs;             // lbm_set_graphs: replay captured two-step graphs
  void* graphs;               // StepGraphs (lbm_capi.cu), created on first use
  void* sc_buf;               // shock capturing: prims (2-D), visc, work planes
  int t64;                    // FP64 temperature inversion in the FP32 / FP16-deviation kernels
};

// Programmatic serialisation of dependent launches: a kernel may be set up, and its
// blocks started, while the launch before it on the stream drains.  Such a kernel
// waits for that launch's results before its first access to memory.  (Launched in
// another way, the wait returns at once.)
// Every kernel of a step is launched so: the gaps between launches were 2 to 6 us of
// a step (channel of 100x24x20, FP64: 136 -> 128 us; 91x75x53: 77.0 -> 69.4; shock of
// 384x128x128: 1162 -> 1136; 256^3 FP32 1943 -> 1921).  None of them lets the next
// launch start early (griddepcontrol.launch_dependents): blocks that only wait then
// take the room of the last blocks at work, and fall on the multiprocessors
// unevenly (256^3 2150 us, the channel 163 us; 800x800 45.3 -> 47.6 us).
__device__ __forceinline__ void wait_previous_launch() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void allow_next_launch() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

// a launch of a kernel that calls wait_previous_launch
template <class... P, class... A>
inline cudaError_t launch_overlapped(void (*kern)(P...), dim3 grid, unsigned block, size_t smem, cudaStream_t st,
                                     A... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = dim3(block);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute attr = {};
  attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr.val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = &attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kern, P(args)...);
}

// Dynamic shared memory of a kernel that may pass 48 KB, and the blocks of it that
// the device holds at once, found on first use.  Internal linkage, as the kernel
// template's own launch stub has it: each translation unit prepares the kernel it
// launches (one prepared flag for all of them left the others' copies at 48 KB).
template <auto kern> static int prepared_blocks(int threads, size_t smem) {
  static const int blocks = [threads, smem] {
    cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, int(smem));
    int n = 1, dev = 0, sms = 1;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, kern, threads, smem);
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    return (n > 1 ? n : 1) * sms;
  }();
  return blocks;
}

struct Batch;

// Per (D, precision) kernel set.
struct Ops {
  // state[i] at every padded node from FP64 device fields (interior layout)
  void (*init)(Handle& h, const double* rho, const double* u, const double* T);
  // one step: pop[cur] -> pop[cur^1] (including the ghost fill)
  void (*step)(Handle& h, const void* src, void* dst);
  void (*step_multipass)(Handle& h, const void* src, void* dst);
  // macroscopic FP64 fields of pop[cur] into device outputs (any may be NULL);
  // totals (device, D+2 doubles) when non-NULL
  void (*macro)(Handle& h, const void* src, double* rho, double* u, double* T, double* totals);
  // time the step's candidates, keep the fastest; returns its index
  int (*autotune)(Handle& h, int reps, float* best_ms);
  // batches: number of tile shapes; build the device instance table and the
  // sorted work list of shape cfg; enqueue one batched step from `parity`
  int (*batch_ncfg)();
  int (*batch_prepare)(Batch& b, int cfg);
  void (*batch_enqueue)(Batch& b, int parity);
  // number of candidates of the step (indices of lbm_set_tile / lbm_autotune)
  int (*ntiles)();
};

// A batch of instances stepped together (lbm_batch_* in include/lbm.h).
struct Batch {
  int n, D, Q, precision;
  Handle** inst;              // one handle per instance (own buffers and scratch)
  void* d_insts;              // device table of BatchInstance (2-D) or SplitInstance (3-D)
  void* d_items;              // device work list of BatchItem or SplitItem, largest instances first
  int nitems;
  int* d_n1rows;              // first global row of each instance's shock capturing (n + 1 entries)
  unsigned ghost_blocks;      // blocks per instance of the batched ghost fill
  int n1rows;                 // rows with shock capturing over all instances (0: none)
  int graph_launches;         // kernel launches of one step's graph
  int tuning;                 // graphs for timing tile shapes: no shock-capturing stencils (they would
                              // overwrite the coefficients the next real step reads)
  int group[10];              // 3-D: first work item of each launch of the step, and their end
  unsigned* d_errs;           // status word per instance
  unsigned* h_errs;           // pinned copy
  cudaStream_t stream;
  int own_stream;
  int cur;                    // parity of the current state (same for all instances)
  int tile_cfg;
  cudaGraphExec_t graph[2];   // one step from parity 0 / 1
  int graph_ready;
  int unstable;
  int unchecked;              // steps enqueued since the status words were last read
  long long launches;
};

// Bounds-check builds (-DLBM_BOUNDS_CHECK) count the population accesses that
// fall outside the handle's buffers in one device counter per translation
// unit; each unit registers a reader of its counter here (a static
// initialiser), and lbm_debug_bounds_violations sums them.
void register_oob_reader(unsigned long long (*reader)());

// Device allocation of the library: cudaMalloc, except that the allocation
// chosen by lbm_debug_fail_alloc fails with cudaErrorMemoryAllocation (and
// allocates nothing), so that tests can take every out-of-memory path.
cudaError_t dev_malloc(void** p, size_t bytes);
template <class T> inline cudaError_t dev_malloc(T** p, size_t bytes) {
  return dev_malloc(reinterpret_cast<void**>(p), bytes);
}

// the opaque handle type of the C interface
}  // namespace lbm
struct lbm_s : public lbm::Handle {};
struct lbm_batch_s : public lbm::Batch {};
namespace lbm {

const Ops* ops_d2_fp64();
const Ops* ops_d2_fp32();
const Ops* ops_d3_fp64();
const Ops* ops_d3_fp32();
const Ops* ops_d2_fp16();
const Ops* ops_d3_fp16();
// step and autotuner with the learned closure (FP32 storage)
void step_d2_fp32_mlp(Handle& h, const void* src, void* dst);
void step_d3_fp32_mlp(Handle& h, const void* src, void* dst);
// exact Peng-Robinson closure (lbm_eos.kind LBM_EOS_PR): step and its autotuner
void step_d2_fp32_pr(Handle& h, const void* src, void* dst);
void step_d3_fp32_pr(Handle& h, const void* src, void* dst);
void step_d2_fp64_pr(Handle& h, const void* src, void* dst);
void step_d3_fp64_pr(Handle& h, const void* src, void* dst);
int autotune_d2_fp32_pr(Handle& h, int reps, float* best_ms);
int autotune_d3_fp32_pr(Handle& h, int reps, float* best_ms);
int autotune_d2_fp64_pr(Handle& h, int reps, float* best_ms);
int autotune_d3_fp64_pr(Handle& h, int reps, float* best_ms);
int autotune_d2_fp32_mlp(Handle& h, int reps, float* best_ms);
int autotune_d3_fp32_mlp(Handle& h, int reps, float* best_ms);
int ntiles_d2_fp32_pr();
int ntiles_d3_fp32_pr();
int ntiles_d2_fp64_pr();
int ntiles_d3_fp64_pr();
int ntiles_d2_fp32_mlp();
int ntiles_d3_fp32_mlp();
// FP32 arithmetic with the FP64 temperature inversion (exact closures):
// step, autotuner and candidate count of FP32 and FP16-deviation storage,
// van der Waals and Peng-Robinson
void step_d2_fp32_t64(Handle& h, const void* src, void* dst);
void step_d3_fp32_t64(Handle& h, const void* src, void* dst);
void step_d2_fp16_t64(Handle& h, const void* src, void* dst);
void step_d3_fp16_t64(Handle& h, const void* src, void* dst);
void step_d2_fp32_pr_t64(Handle& h, const void* src, void* dst);
void step_d3_fp32_pr_t64(Handle& h, const void* src, void* dst);
int autotune_d2_fp32_t64(Handle& h, int reps, float* best_ms);
int autotune_d3_fp32_t64(Handle& h, int reps, float* best_ms);
int autotune_d2_fp16_t64(Handle& h, int reps, float* best_ms);
int autotune_d3_fp16_t64(Handle& h, int reps, float* best_ms);
int autotune_d2_fp32_pr_t64(Handle& h, int reps, float* best_ms);
int autotune_d3_fp32_pr_t64(Handle& h, int reps, float* best_ms);
int ntiles_d2_fp32_t64();
int ntiles_d3_fp32_t64();
int ntiles_d2_fp16_t64();
int ntiles_d3_fp16_t64();
int ntiles_d2_fp32_pr_t64();
int ntiles_d3_fp32_pr_t64();

}  // namespace lbm
