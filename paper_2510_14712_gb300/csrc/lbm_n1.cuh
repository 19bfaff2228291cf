// lbm_n1.cuh - shock-capturing numerical transport coefficients (Sec. 4.4,
// Eqs. shock_cap and shock_cap_k), computed after each step from that step's
// primitive fields and used by the next step's collision:
//
//   {mu, eta}^num = rho C_{mu,eta} F(|grad^4 S|),  k^num = rho c_s C_k F(|grad^4 |grad s||)
//
// with S = |grad u + grad u^T| / 2, grad s = (c_v/T) grad T - R/(rho (1 - b rho)) grad rho
// (van der Waals; the general identity for Peng-Robinson), |grad^4 f| =
// sqrt(sum_a (d_a^4 f)^2) over the per-axis five-point fourth differences
// (r = 5, delta x^(r+1) = 1), F the separable binomial filter (1, 4, 6, 4, 1)/16
// along every axis, c_s the fluid's sound speed at (rho, T).  Neighbours wrap
// on periodic axes and are clamped to the nearest interior node on
// non-periodic x faces.  Fields live on the padded plane layout of the handle
// (offset (z Ny + y) pitch + x + G, one plane per component).  Three forms
// share the per-node arithmetic: in 2-D the step itself leaves S and |grad s|
// (its block holds the neighbours' u, T and rho) and one launch over tiles does
// the rest; in 3-D one launch for S and |grad s| and one over columns of
// the box (3-D batches: the same over the blocks of every instance); one block per row
// for the 2-D batches.
#pragma once

#include "lbm_tile2d.cuh"

namespace lbm {

// v mod n for a shift of at most a few nodes: one comparison in range
__device__ __forceinline__ int n1_wrap(int v, int n) { return unsigned(v) < unsigned(n) ? v : modp(v, n); }

// Values a stage computes at one node, stored to K planes of its output.
template <typename real, int K> struct N1Vals {
  real v[K];
};

template <typename real, int K>
__device__ __forceinline__ void n1_store(const Params& p, real* out, unsigned o, const N1Vals<real, K>& r) {
#pragma unroll
  for (int k = 0; k < K; ++k) out[k * p.plane + o] = r.v[k];
}

// offset of the interior neighbour (x, y, z) + s e_a of the node at offset o:
// wrapped on periodic axes, clamped to the nearest interior node on a
// non-periodic x
__device__ __forceinline__ unsigned n1_nb(const Params& p, int x, int y, int z, unsigned o, int a, int s) {
  if (a == 0) {
    int xs = x + s;
    xs = p.periodic_x ? n1_wrap(xs, p.Nx) : (xs < 0 ? 0 : (xs >= p.Nx ? p.Nx - 1 : xs));
    return o + unsigned(xs - x);
  }
  if (a == 1) return o + unsigned((n1_wrap(y + s, p.Ny) - y) * p.pitch);
  return o + unsigned((n1_wrap(z + s, p.Nz) - z) * p.Ny * p.pitch);
}

// ---- per-node stages (shared by the single-instance and batched kernels) ----
// No stage reads a buffer it writes, so every input goes through the read-only
// path (__ldg).  Each returns its values; the caller stores them.

template <typename real> __device__ __forceinline__ real n1_ld(const real* q) { return __ldg(q); }

// five-point fourth difference and binomial (1, 4, 6, 4, 1)/16 of the values at
// offsets -2 .. +2 along one axis, and the coefficients from the filtered norms
// (one definition for every form; V: a scalar or a packed pair, multiply-adds
// written out, so that the forms give the same bits)
template <typename V> __device__ __forceinline__ V n1_fourth(V vm2, V vm1, V v0, V vp1, V vp2) {
  return mad(V(-4), vp1 + vm1, mad(V(6), v0, vp2 + vm2));
}
template <typename V> __device__ __forceinline__ V n1_binom5(V vm2, V vm1, V v0, V vp1, V vp2) {
  return mad(V(4), vp1 + vm1, mad(V(6), v0, vp2 + vm2)) * V(0.0625f);
}
// c_s of k^num
template <typename real> __device__ __forceinline__ real n1_sound(const Model<real>& m, real r, real t) {
  return root(positive(eos_cs2(m, r, t)));
}
__device__ __forceinline__ F2 n1_sound(const Model<float>& m, F2 r, F2 t) {
  return m.kind == LBM_EOS_PR ? F2(n1_sound(m, r.x, t.x), n1_sound(m, r.y, t.y)) : root(positive(vdw_cs2(m, r, t)));
}
template <typename real, typename V>
__device__ __forceinline__ N1Vals<V, 3> n1_coefs(const Params& p, const Model<real>& m, V r, V t, V s4, V g4) {
  const V cs = n1_sound(m, r, t);
  return {{r * V(real(p.sc_c[0])) * s4, r * V(real(p.sc_c[1])) * s4, r * cs * V(real(p.sc_c[2])) * g4}};
}

// S and |grad s| at the node
template <int D, typename real>
__device__ __forceinline__ N1Vals<real, 2> n1_strain_at(const Params& p, const real* __restrict__ rho,
                                                        const real* __restrict__ u, const real* __restrict__ T,
                                                        int x, int y, int z, unsigned o) {
  unsigned op[D], om[D];
#pragma unroll
  for (int a = 0; a < D; ++a) {
    op[a] = n1_nb(p, x, y, z, o, a, 1);
    om[a] = n1_nb(p, x, y, z, o, a, -1);
  }
  real g[D][D];                                    // g[a][b] = d_a u_b (central)
#pragma unroll
  for (int a = 0; a < D; ++a)
#pragma unroll
    for (int b = 0; b < D; ++b)
      g[a][b] = real(0.5) * (n1_ld(u + b * p.plane + op[a]) - n1_ld(u + b * p.plane + om[a]));
  real gT[D], gr[D];
#pragma unroll
  for (int a = 0; a < D; ++a) {
    gT[a] = real(0.5) * (n1_ld(T + op[a]) - n1_ld(T + om[a]));
    gr[a] = real(0.5) * (n1_ld(rho + op[a]) - n1_ld(rho + om[a]));
  }
  N1Vals<real, 2> v;
  n1_norms<D>(model_of<real>(p), g, gT, gr, n1_ld(rho + o), n1_ld(T + o), v.v[0], v.v[1]);
  return v;
}

// norm of the per-axis fourth differences of the two fields of `in` at the node (2-D)
template <typename real>
__device__ __forceinline__ N1Vals<real, 2> n1_d4_at(const Params& p, const real* __restrict__ in, int x, int y, unsigned o) {
  unsigned nb[2][4];                               // offsets of the -2, -1, +1, +2 neighbours along a
#pragma unroll
  for (int a = 0; a < 2; ++a) {
    nb[a][0] = n1_nb(p, x, y, 0, o, a, -2);
    nb[a][1] = n1_nb(p, x, y, 0, o, a, -1);
    nb[a][2] = n1_nb(p, x, y, 0, o, a, 1);
    nb[a][3] = n1_nb(p, x, y, 0, o, a, 2);
  }
  N1Vals<real, 2> res;
#pragma unroll
  for (int f = 0; f < 2; ++f) {
    const real* v = in + f * p.plane;
    real acc = real(0);
#pragma unroll
    for (int a = 0; a < 2; ++a) {
      const real d4 = n1_fourth(n1_ld(v + nb[a][0]), n1_ld(v + nb[a][1]), n1_ld(v + o), n1_ld(v + nb[a][2]),
                                n1_ld(v + nb[a][3]));
      acc = mad(d4, d4, acc);
    }
    res.v[f] = root(acc);
  }
  return res;
}

// binomial (1, 4, 6, 4, 1)/16 along axis a of both fields of `in` at the node (2-D)
template <typename real>
__device__ __forceinline__ N1Vals<real, 2> n1_filter_at(const Params& p, int a, const real* __restrict__ in, int x, int y,
                                                        unsigned o) {
  const unsigned m2 = n1_nb(p, x, y, 0, o, a, -2), m1 = n1_nb(p, x, y, 0, o, a, -1);
  const unsigned p1 = n1_nb(p, x, y, 0, o, a, 1), p2 = n1_nb(p, x, y, 0, o, a, 2);
  N1Vals<real, 2> res;
#pragma unroll
  for (int f = 0; f < 2; ++f) {
    const real* v = in + f * p.plane;
    res.v[f] = n1_binom5(n1_ld(v + m2), n1_ld(v + m1), n1_ld(v + o), n1_ld(v + p1), n1_ld(v + p2));
  }
  return res;
}

// Buffers of one handle's shock capturing: the step's rho, u (D planes), T (by
// default the 2-D step's copy in sc_prims), the coefficients (3 planes) followed by
// the work planes w0, w1 (2 each; w1 in 2-D only).  S and |grad s| go to w0; the tiled
// and column forms go from there to the coefficients, the 2-D batched stages run fourth
// differences w0 -> w1, the x pass w1 -> w0, the y pass with the coefficients.
template <int D, typename real> struct N1Buffers {
  const real *rho, *u, *T;
  real *visc, *w0, *w1;
  __host__ __device__ N1Buffers(const Params& p, const real* rho_, const real* u_, const real* T_)
      : rho(rho_), u(u_), T(T_) {
    visc = static_cast<real*>(const_cast<void*>(p.sc_visc));
    w0 = visc + 3 * p.plane;
    w1 = w0 + 2 * p.plane;
  }
  __host__ __device__ explicit N1Buffers(const Params& p)
      : N1Buffers(p, static_cast<const real*>(p.sc_prims), static_cast<const real*>(p.sc_prims) + p.plane,
                  static_cast<const real*>(p.sc_prims) + (1 + D) * p.plane) {}
};

// ---- single-instance kernels ----

// 3-D: S and |grad s|, one unit of nodes per thread: the loads along y and z and the
// arithmetic serve both nodes of an FP32 unit (one node per thread, 64 scalar loads
// for two nodes: 84 us at 384x128x128, now 53 us).
template <typename S, typename real>
__device__ __forceinline__ void n1_strain_units(const Params& p, unsigned n, FastDiv dnx, FastDiv dny, const real* __restrict__ rho,
                                                 const real* __restrict__ u, const real* __restrict__ T, const unsigned block) {
  using U = Unit<S, real>;
  using V = typename U::V;
  constexpr int N = U::N;
  const unsigned gid = block * 128u + threadIdx.x;
  if (gid >= n) return;
  const unsigned row = dnx.div(gid), z = dny.div(row);
  const int y = int(row - z * unsigned(p.Ny)), x = N * int(gid - row * unsigned((p.Nx + N - 1) / N));
  const bool whole = x + N <= p.Nx;                              // every node of the unit is one of the box
  const unsigned o = row * unsigned(p.pitch) + unsigned(x + p.G);
  const unsigned xm = n1_nb(p, x, y, int(z), o, 0, -1), xp = n1_nb(p, x, y, int(z), o, 0, whole ? N : 1);
  const unsigned nb[2][2] = {{n1_nb(p, x, y, int(z), o, 1, -1), n1_nb(p, x, y, int(z), o, 1, 1)},
                             {n1_nb(p, x, y, int(z), o, 2, -1), n1_nb(p, x, y, int(z), o, 2, 1)}};
  auto differences = [&](const real* f, V& c, V& dx, V& dy, V& dz) {
    const V half = V(real(0.5));
    c = U::ld_field(f + o);
    const real l = n1_ld(f + xm), r = n1_ld(f + xp);
    V up, um;
#pragma unroll
    for (int k = 0; k < N; ++k) {
      U::set(up, k, whole && k + 1 < N ? U::get(c, (k + 1) % N) : r);
      U::set(um, k, k > 0 ? U::get(c, k > 0 ? k - 1 : 0) : l);
    }
    dx = half * (up - um);
    dy = half * (U::ld_field(f + nb[0][1]) - U::ld_field(f + nb[0][0]));
    dz = half * (U::ld_field(f + nb[1][1]) - U::ld_field(f + nb[1][0]));
  };
  V g[3][3], gT[3], gr[3], r, t, c, Sn, gn;
#pragma unroll
  for (int b = 0; b < 3; ++b) differences(u + b * p.plane, c, g[0][b], g[1][b], g[2][b]);
  differences(T, t, gT[0], gT[1], gT[2]);
  differences(rho, r, gr[0], gr[1], gr[2]);
  n1_norms<3>(model_of<real>(p), g, gT, gr, r, t, Sn, gn);
  const N1Buffers<3, real> b(p);
  U::store_field(b.w0 + o, Sn, whole);
  U::store_field(b.w0 + p.plane + o, gn, whole);
}
template <typename S, typename real>
__global__ void __launch_bounds__(128)
k_n1_strain_3d(const __grid_constant__ Params p, unsigned n, FastDiv dnx, FastDiv dny, const real* __restrict__ rho,
               const real* __restrict__ u, const real* __restrict__ T) {
  wait_previous_launch();
  n1_strain_units<S, real>(p, n, dnx, dny, rho, u, T, blockIdx.x);
}

// ---- 2-D single-instance form: one launch over tiles of the plane ----
// The step's blocks leave S and |grad s| in w0 (n1_norms on the fields they hold
// in shared memory), rho and T in sc_prims.  A block here owns 64 x 16 nodes (one
// unit of Unit<> per thread and step): S and |grad s| of the tile and a four-node
// halo, the norm of their fourth differences on a two-node halo, the x pass on
// the tile's columns and a two-row halo, the y pass with the coefficients.  Halo
// positions take the values of the node the row-mapped stencils read there:
// wrapped on a periodic axis, clamped to the nearest interior node otherwise.
// Two tiled launches that read the fields again (strain with fourth differences,
// filter with coefficients; 48 registers, one node per thread and pass, 572
// instructions per node) took 137 + 107 us at 4096x2048; this launch 67 us (85 with
// each load of the box followed by its store).
constexpr int kN1TileX = 64, kN1TileY = 16, kN1Threads = 256;

template <typename S, typename real>
__global__ void __launch_bounds__(kN1Threads) k_n1_coef_2d(const __grid_constant__ Params p, int ntx) {
  wait_previous_launch();
  using U = Unit<S, real>;
  using V = typename U::V;
  constexpr int N = U::N, HX = 4, P4 = kN1TileX + 2 * HX, H4 = kN1TileY + 8, P2 = kN1TileX + 4, H2 = kN1TileY + 4;
  constexpr int PX = kN1TileX;
  __shared__ __align__(16) real s4[2][H4 * P4];          // S, |grad s|; later the x-filtered norms
  __shared__ __align__(16) real s2[2][H2 * P2];          // norms of the fourth differences
  const N1Buffers<2, real> b(p);
  const Model<real> m = model_of<real>(p);
  const int tid = threadIdx.x;
  const int x0 = int(blockIdx.x % unsigned(ntx)) * kN1TileX, y0 = int(blockIdx.x / unsigned(ntx)) * kN1TileY;
  const unsigned pitch = unsigned(p.pitch);
  // node that a stencil reads at x: wrapped, or clamped to the box
  auto src = [&](int x) { return p.periodic_x ? n1_wrap(x, p.Nx) : min(max(x, 0), p.Nx - 1); };
  // units of the box whose nodes are not neighbours in memory, or whose halo is clamped
  const bool edge = x0 < HX || x0 + kN1TileX + HX > p.Nx;
  // every load of the box in flight before the first store
  constexpr int K4 = (P4 / N * H4 + kN1Threads - 1) / kN1Threads;
  V box[2][K4];
#pragma unroll
  for (int i = 0; i < K4; ++i) {
    const int k = min(tid + i * kN1Threads, P4 / N * H4 - 1), r = k / (P4 / N), x = x0 + N * (k - r * (P4 / N)) - HX;
    const unsigned row = unsigned(n1_wrap(y0 + r - 4, p.Ny)) * pitch + unsigned(p.G);
#pragma unroll
    for (int f = 0; f < 2; ++f) {
      const real* w = b.w0 + f * p.plane + row;
      if (!edge) {
        box[f][i] = U::ld_field(w + x);
      } else {
#pragma unroll
        for (int q = 0; q < N; ++q) U::set(box[f][i], q, __ldg(w + src(x + q)));
      }
    }
  }
#pragma unroll
  for (int i = 0; i < K4; ++i)
#pragma unroll
    for (int f = 0; f < 2; ++f)
      if (tid + i * kN1Threads < P4 / N * H4) U::st(s4[f] + N * (tid + i * kN1Threads), box[f][i]);
  __syncthreads();
  for (int k = tid; k < P2 / N * H2; k += kN1Threads) {
    const int r = k / (P2 / N), u = k - r * (P2 / N), x = x0 + N * u - 2;
#pragma unroll
    for (int f = 0; f < 2; ++f) {
      V v;
      if (!edge || p.periodic_x) {
        const real* c = s4[f] + (r + 2) * P4 + N * u + 2;
        V w[5];
        U::five(c, w);
        const V dx = n1_fourth(w[0], w[1], w[2], w[3], w[4]);
        const V dy = n1_fourth(U::ld(c - 2 * P4), U::ld(c - P4), w[2], U::ld(c + P4), U::ld(c + 2 * P4));
        v = root(mad(dy, dy, dx * dx));
      } else {                                            // the norm of the clamped node, one node at a time
#pragma unroll
        for (int q = 0; q < N; ++q) {
          const real* c = s4[f] + (r + 2) * P4 + min(max(src(x + q) - x0 + HX, 2), P4 - 3);
          const real dx = n1_fourth(c[-2], c[-1], c[0], c[1], c[2]);
          const real dy = n1_fourth(c[-2 * P4], c[-P4], c[0], c[P4], c[2 * P4]);
          U::set(v, q, root(mad(dy, dy, dx * dx)));
        }
      }
      U::st(s2[f] + r * P2 + N * u, v);
    }
  }
  __syncthreads();
  for (int k = tid; k < PX / N * H2; k += kN1Threads) {
    const int r = k / (PX / N), u = k - r * (PX / N);
#pragma unroll
    for (int f = 0; f < 2; ++f) {
      const real* c = s2[f] + r * P2 + N * u + 2;
      V w[5];
      U::five(c, w);
      U::st(s4[f] + r * PX + N * u, n1_binom5(w[0], w[1], w[2], w[3], w[4]));
    }
  }
  __syncthreads();
  for (int k = tid; k < PX / N * kN1TileY; k += kN1Threads) {
    const int r = k / (PX / N), u = k - r * (PX / N), x = x0 + N * u, y = y0 + r;
    if (x >= p.Nx || y >= p.Ny) continue;
    V q[2];
#pragma unroll
    for (int f = 0; f < 2; ++f) {
      const real* c = s4[f] + r * PX + N * u;
      q[f] = n1_binom5(U::ld(c), U::ld(c + PX), U::ld(c + 2 * PX), U::ld(c + 3 * PX), U::ld(c + 4 * PX));
    }
    const unsigned o = unsigned(y) * pitch + unsigned(x + p.G);
    const N1Vals<V, 3> res = n1_coefs<real, V>(p, m, U::ld_field(b.rho + o), U::ld_field(b.T + o), q[0], q[1]);
#pragma unroll
    for (int j = 0; j < 3; ++j) U::store_field(b.visc + j * p.plane + o, res.v[j], x + N - 1 < p.Nx);
  }
}

// ---- 3-D single-instance form: one launch from S and |grad s| to the coefficients ----
// A block marches z over a column of TX x TY nodes: S and |grad s| of five planes
// with a four-node halo in the plane, in a ring of shared memory; the norm of the
// fourth differences of the ring's middle plane on a two-node halo, its x pass, its
// y pass at the nodes, and the z pass over five planes held in registers.  The next
// plane is requested before this one is worked on; three barriers per plane.  Halo
// positions as in the 2-D form, which gives the bits of the row-mapped stages.
// Those (fourth differences, two filter passes, last pass with the coefficients:
// four launches with a pass over memory each) took 193 us at 384x128x128 in FP32, this
// launch 151.
template <typename S, typename real> struct N1Column {
  using U = Unit<S, real>;
  static constexpr int N = U::N, TX = 32 * N, TY = 8, HX = 4;
  static constexpr int P4 = TX + 2 * HX, H4 = TY + 8, P2 = TX + 4, H2 = TY + 4, NU = TY * 32 / kN1Threads;
  static constexpr int kPlane = H4 * P4;                         // one field of one plane
  static constexpr size_t kBytes = sizeof(real) * 2 * (5 * kPlane + H2 * P2 + H2 * TX);
};
// the arguments of one column: of a handle, here, or of an instance of a batch
template <typename real> struct N1CoefArgs {
  const Params& p;
  const real *rho, *T;
  int ntx, nty, nseg;
  unsigned block;
};
template <typename real> struct N1CoefHandle {
  Params p;
  const real *rho, *T;
  int ntx, nty, nseg;
  __device__ __forceinline__ N1CoefArgs<real> args() const { return {p, rho, T, ntx, nty, nseg, blockIdx.x}; }
};
// (the body stands in the kernel: in a function that a kernel of each calls the compiler
// took 114 registers instead of 80, and bounded to 85 the column took 158 us for 152)
template <typename S, typename real, class Src>
__global__ void __launch_bounds__(kN1Threads) k_n1_coef_3d(const __grid_constant__ Src from) {
  wait_previous_launch();
  const N1CoefArgs<real> arg = from.args();
  const Params& p = arg.p;
  const int ntx = arg.ntx, nty = arg.nty, nseg = arg.nseg;
  using C = N1Column<S, real>;
  using U = typename C::U;
  using V = typename U::V;
  constexpr int N = U::N, P4 = C::P4, P2 = C::P2, H2 = C::H2, TX = C::TX, HX = C::HX, NU = C::NU;
  constexpr int U4 = P4 / N, K4 = (U4 * C::H4 + kN1Threads - 1) / kN1Threads;
  extern __shared__ __align__(128) unsigned char smem_raw[];
  real* ring = reinterpret_cast<real*>(smem_raw);
  real* s2 = ring + 10 * C::kPlane;                              // norms of the fourth differences
  real* sx = s2 + 2 * H2 * P2;                                   // the same after the x pass
  const N1Buffers<3, real> b(p, arg.rho, nullptr, arg.T);
  const Model<real> m = model_of<real>(p);
  const int tid = threadIdx.x;
  int blk = int(arg.block);
  const int x0 = (blk % ntx) * TX;
  blk /= ntx;
  const int y0 = (blk % nty) * C::TY, seg = blk / nty;
  const int mb = int((long long)p.Nz * seg / nseg), me = int((long long)p.Nz * (seg + 1) / nseg);
  const unsigned pitch = unsigned(p.pitch), zs = unsigned(p.Ny) * pitch, ztop = zs * unsigned(p.Nz);
  // node that a stencil reads at x: wrapped, or clamped to the box
  auto src = [&](int x) { return p.periodic_x ? n1_wrap(x, p.Nx) : min(max(x, 0), p.Nx - 1); };
  const bool edge = x0 < HX || x0 + TX + HX > p.Nx;
  unsigned at[K4][N];                                            // in-plane offsets of this thread's box units
#pragma unroll
  for (int k = 0; k < K4; ++k) {
    const int q = min(tid + k * kN1Threads, U4 * C::H4 - 1), r = q / U4, x = x0 + N * (q - r * U4) - HX;
    const unsigned row = unsigned(n1_wrap(y0 + r - 4, p.Ny)) * pitch + unsigned(p.G);
#pragma unroll
    for (int j = 0; j < N; ++j) at[k][j] = row + unsigned(src(x + j));
  }
  unsigned zl = unsigned(n1_wrap(mb - 4, p.Nz)) * zs;            // plane to load next
  V nxt[2][K4];
  auto load = [&] {
#pragma unroll
    for (int f = 0; f < 2; ++f) {
      const real* w = b.w0 + f * p.plane + zl;
#pragma unroll
      for (int k = 0; k < K4; ++k) {
        if (!edge) {
          nxt[f][k] = U::ld_field(w + at[k][0]);
        } else {
#pragma unroll
          for (int j = 0; j < N; ++j) U::set(nxt[f][k], j, __ldg(w + at[k][j]));
        }
      }
    }
    zl = zl + zs == ztop ? 0u : zl + zs;
  };
  load();
  const int ux = tid % 32, uy = tid / 32, x = x0 + N * ux;
  V zr[NU][2][5];                                                // x- and y-filtered norms of five planes
#pragma unroll
  for (int i = 0; i < NU; ++i)
#pragma unroll
    for (int f = 0; f < 2; ++f)
#pragma unroll
      for (int k = 0; k < 5; ++k) zr[i][f][k] = V(0);
  unsigned zo = unsigned(mb) * zs;                               // plane of the next output
  int slot = 0;                                                  // ring slot of plane pl
  for (int pl = mb - 4; pl <= me + 3; ++pl) {
    real* now = ring + slot * 2 * C::kPlane;
#pragma unroll
    for (int f = 0; f < 2; ++f)
#pragma unroll
      for (int k = 0; k < K4; ++k)
        if (tid + k * kN1Threads < U4 * C::H4) U::st(now + f * C::kPlane + N * (tid + k * kN1Threads), nxt[f][k]);
    if (pl < me + 3) load();
    __syncthreads();
    const int cur = slot;
    slot = slot == 4 ? 0 : slot + 1;
    if (pl < mb) continue;
    auto plane = [&](const int d) {                              // ring slot of plane pl - 2 + d
      const int q = cur + 3 + d;                                 // cur - 2 + d + 5
      return ring + (q >= 5 ? q - 5 : q) * 2 * C::kPlane;
    };
    const real *cm2 = plane(-2), *cm1 = plane(-1), *c0 = plane(0), *cp1 = plane(1), *cp2 = plane(2);
    for (int k = tid; k < P2 / N * H2; k += kN1Threads) {
      const int r = k / (P2 / N), u = k - r * (P2 / N);
#pragma unroll
      for (int f = 0; f < 2; ++f) {
        V v;
        if (!edge || p.periodic_x) {
          const int c = f * C::kPlane + (r + 2) * P4 + N * u + 2;
          const real* q = c0 + c;
          V w[5];
          U::five(q, w);
          const V dx = n1_fourth(w[0], w[1], w[2], w[3], w[4]);
          const V dy = n1_fourth(U::ld(q - 2 * P4), U::ld(q - P4), w[2], U::ld(q + P4), U::ld(q + 2 * P4));
          const V dz = n1_fourth(U::ld(cm2 + c), U::ld(cm1 + c), w[2], U::ld(cp1 + c), U::ld(cp2 + c));
          v = root(mad(dz, dz, mad(dy, dy, dx * dx)));
        } else {                                                 // the norm of the clamped node, one node at a time
#pragma unroll
          for (int j = 0; j < N; ++j) {
            const int xc = min(max(src(x0 + N * u - 2 + j) - x0 + HX, 2), P4 - 3);
            const int c = f * C::kPlane + (r + 2) * P4 + xc;
            const real* q = c0 + c;
            const real dx = n1_fourth(q[-2], q[-1], q[0], q[1], q[2]);
            const real dy = n1_fourth(q[-2 * P4], q[-P4], q[0], q[P4], q[2 * P4]);
            const real dz = n1_fourth(cm2[c], cm1[c], q[0], cp1[c], cp2[c]);
            U::set(v, j, root(mad(dz, dz, mad(dy, dy, dx * dx))));
          }
        }
        U::st(s2 + f * H2 * P2 + r * P2 + N * u, v);
      }
    }
    __syncthreads();
    for (int k = tid; k < 32 * H2; k += kN1Threads) {
      const int r = k / 32, u = k % 32;
#pragma unroll
      for (int f = 0; f < 2; ++f) {
        const real* c = s2 + f * H2 * P2 + r * P2 + N * u + 2;
        V w[5];
        U::five(c, w);
        U::st(sx + f * H2 * TX + r * TX + N * u, n1_binom5(w[0], w[1], w[2], w[3], w[4]));
      }
    }
    __syncthreads();
#pragma unroll
    for (int i = 0; i < NU; ++i) {
      const int r = uy + i * (kN1Threads / 32), y = y0 + r;
      V q[2];
#pragma unroll
      for (int f = 0; f < 2; ++f) {
        const real* c = sx + f * H2 * TX + r * TX + N * ux;
        V* z = zr[i][f];
#pragma unroll
        for (int k = 0; k < 4; ++k) z[k] = z[k + 1];
        z[4] = n1_binom5(U::ld(c), U::ld(c + TX), U::ld(c + 2 * TX), U::ld(c + 3 * TX), U::ld(c + 4 * TX));
        q[f] = n1_binom5(z[0], z[1], z[2], z[3], z[4]);
      }
      if (pl < mb + 4 || x >= p.Nx || y >= p.Ny) continue;
      const unsigned o = zo + unsigned(y) * pitch + unsigned(x + p.G);
      const N1Vals<V, 3> res = n1_coefs<real, V>(p, m, U::ld_field(b.rho + o), U::ld_field(b.T + o), q[0], q[1]);
#pragma unroll
      for (int j = 0; j < 3; ++j) U::store_field(b.visc + j * p.plane + o, res.v[j], x + N - 1 < p.Nx);
    }
    if (pl >= mb + 4) zo += zs;
  }
}

// S and |grad s| of a plane from its rho, u, T, which also go to sc_prims (the
// multi-pass step keeps them in its scratch area)
template <typename real>
__global__ void __launch_bounds__(256) k_n1_norms_2d(const __grid_constant__ Params p, const real* __restrict__ rho,
                                                     const real* __restrict__ u, const real* __restrict__ T) {
  wait_previous_launch();
  const long long n = blockIdx.x * 256LL + threadIdx.x;
  if (n >= (long long)p.Nx * p.Ny) return;
  const int y = int(n / p.Nx), x = int(n - (long long)y * p.Nx);
  const unsigned o = unsigned(y) * unsigned(p.pitch) + unsigned(x + p.G);
  const N1Buffers<2, real> b(p);
  n1_store(p, b.w0, o, n1_strain_at<2, real>(p, rho, u, T, x, y, 0, o));
  const_cast<real*>(b.rho)[o] = rho[o];
  const_cast<real*>(b.T)[o] = T[o];
}

// z-segments of the coefficient columns: whole rounds of resident blocks over all
// columns of the launch against the eight planes (two thirds of a plane's work) that
// each segment repeats
inline int n1_segments(const Params& p, int slots, long long columns) {
  int nseg = 1;
  long long least = -1;
  for (int k = 1; k <= std::min(p.Nz, 32); ++k) {
    const long long cost = (columns * k + slots - 1) / slots * ((p.Nz + k - 1) / k + 5);
    if (least < 0 || cost < least) {
      least = cost;
      nseg = k;
    }
  }
  return nseg;
}

// The whole update of a handle's coefficients.  2-D: one launch after a step that
// left S and |grad s| (`rho` null), two after one that left rho, u (D planes) and
// T; 3-D: two from rho, u, T (padded plane layout).
template <int D, typename S, typename real>
inline int n1_update(const Params& p, cudaStream_t st, const real* rho, const real* u, const real* T) {
  if constexpr (D == 2) {
    if (rho) launch_overlapped(k_n1_norms_2d<real>, dim3(unsigned(((long long)p.Nx * p.Ny + 255) / 256)), 256, 0, st, p, rho, u, T);
    const int ntx = (p.Nx + kN1TileX - 1) / kN1TileX, nty = (p.Ny + kN1TileY - 1) / kN1TileY;
    launch_overlapped(k_n1_coef_2d<S, real>, dim3(unsigned(ntx) * unsigned(nty)), kN1Threads, 0, st, p, ntx);
    return rho ? 2 : 1;
  } else {
    using C = N1Column<S, real>;
    using Src = N1CoefHandle<real>;
    const int slots = prepared_blocks<k_n1_coef_3d<S, real, Src>>(kN1Threads, C::kBytes);
    const unsigned nx = unsigned((p.Nx + C::N - 1) / C::N), n = nx * unsigned(p.Ny) * unsigned(p.Nz);
    launch_overlapped(k_n1_strain_3d<S, real>, dim3((n + 127u) / 128u), 128, 0, st, p, n, FastDiv(nx),
                      FastDiv(unsigned(p.Ny)), rho, u, T);
    const int ntx = (p.Nx + C::TX - 1) / C::TX, nty = (p.Ny + C::TY - 1) / C::TY, nseg = n1_segments(p, slots, (long long)ntx * nty);
    launch_overlapped(k_n1_coef_3d<S, real, Src>, dim3(unsigned(ntx) * unsigned(nty) * unsigned(nseg)), kN1Threads, C::kBytes,
                      st, Src{p, rho, T, ntx, nty, nseg});
    return 2;
  }
}

// ---- batched kernels: one block per row of every instance with shock capturing ----

// rowstart[k] = first global row of instance k (prefix sum of Ny Nz over the
// instances with shock capturing on, 0 rows for the others); rowstart[n] = total
__device__ __forceinline__ int n1_instance(const int* __restrict__ rowstart, int n, int row) {
  int lo = 0, hi = n;                              // largest k < n with rowstart[k] <= row
  while (hi - lo > 1) {
    const int mid = (lo + hi) >> 1;
    if (rowstart[mid] <= row) lo = mid;
    else hi = mid;
  }
  return lo;
}

// stage 0: S and |grad s|, 1: fourth differences, 2: x pass, 3: y pass and coefficients
template <typename real, int STAGE>
__global__ void k_n1_batch(const BatchInstance* __restrict__ insts, const int* __restrict__ rowstart, int n) {
  wait_previous_launch();
  const int k = n1_instance(rowstart, n, blockIdx.x);
  const Params& p = insts[k].p;
  const N1Buffers<2, real> b(p);
  const int y = blockIdx.x - rowstart[k];
  const Model<real> m = model_of<real>(p);
  for (int x = threadIdx.x; x < p.Nx; x += blockDim.x) {
    const unsigned o = unsigned(y) * unsigned(p.pitch) + unsigned(x + p.G);
    if constexpr (STAGE == 0) n1_store(p, b.w0, o, n1_strain_at<2, real>(p, b.rho, b.u, b.T, x, y, 0, o));
    else if constexpr (STAGE == 1) n1_store(p, b.w1, o, n1_d4_at(p, static_cast<const real*>(b.w0), x, y, o));
    else if constexpr (STAGE == 2) n1_store(p, b.w0, o, n1_filter_at(p, 0, static_cast<const real*>(b.w1), x, y, o));
    else {
      const N1Vals<real, 2> q = n1_filter_at(p, 1, static_cast<const real*>(b.w0), x, y, o);
      n1_store(p, b.visc, o, n1_coefs(p, m, n1_ld(b.rho + o), n1_ld(b.T + o), q.v[0], q.v[1]));
    }
  }
}

// the update of every 2-D instance with shock capturing on: four launches over `rows`
// global rows
template <typename real>
inline int n1_update_batch(const BatchInstance* insts, const int* rowstart, int n, int rows, cudaStream_t st) {
  launch_overlapped(k_n1_batch<real, 0>, dim3(unsigned(rows)), 128u, 0, st, insts, rowstart, n);
  launch_overlapped(k_n1_batch<real, 1>, dim3(unsigned(rows)), 128u, 0, st, insts, rowstart, n);
  launch_overlapped(k_n1_batch<real, 2>, dim3(unsigned(rows)), 128u, 0, st, insts, rowstart, n);
  launch_overlapped(k_n1_batch<real, 3>, dim3(unsigned(rows)), 128u, 0, st, insts, rowstart, n);
  return 4;
}

}  // namespace lbm
