// lbm_kernels.cuh - kernels of the library, templated on the dimension D,
// the storage type of the populations and the arithmetic type.
//
// Data layout in HBM (all kernels):
//   population p_i of node (x, y, z) at  base + i*plane + (z*Ny + y)*pitch + (x + G)
//   with G = 4 ghost layers per non-periodic x face (G = 0 when x is
//   periodic), pitch >= Nx + 2G rounded up to 32 elements, plane = Nz*Ny*pitch.
//   The buffer holds the post-collision populations of the last step (pull
//   scheme: node x reads p_i at x - c_i).
//
// The split step (this file) is: moments -> primitive fields -> collide, with the
// ghost layers filled by the collision or, at walls, by a launch of their own.  It
// keeps the moment and primitive fields of every node in the handle's scratch
// planes.  3-D boxes step so; 2-D planes take one tile per block (lbm_tile2d.cuh),
// or this form when the multi-pass step is asked for.
#pragma once

#include "lbm_internal.cuh"
#include "lbm_mlp_tc.cuh"

namespace lbm {

// ---------------------------------------------------------------------------
// storage traits: how one population value is kept in HBM
// ---------------------------------------------------------------------------
struct Fp16Dev {};  // tag: FP16 storage of p_i - p_i^ref

template <typename S> struct Store;
// ld/st: plain; ld_last: last read of the value in this step (evict-first);
// st_stream: streaming store of the new populations (evict-first).
template <> struct Store<double> {
  using T = double;
  template <typename real, typename I> __device__ static real ld(const T* p, I o, float) { return real(__ldg(p + o)); }
  template <typename real, typename I> __device__ static real ld_last(const T* p, I o, float) { return real(__ldcs(p + o)); }
  template <typename real, typename I> __device__ static void st(T* p, I o, real v, float) { p[o] = double(v); }
  template <typename real, typename I> __device__ static void st_stream(T* p, I o, real v, float) { __stcs(p + o, double(v)); }
};
template <> struct Store<float> {
  using T = float;
  template <typename real, typename I> __device__ static real ld(const T* p, I o, float) { return real(__ldg(p + o)); }
  template <typename real, typename I> __device__ static real ld_last(const T* p, I o, float) { return real(__ldcs(p + o)); }
  template <typename real, typename I> __device__ static void st(T* p, I o, real v, float) { p[o] = float(v); }
  template <typename real, typename I> __device__ static void st_stream(T* p, I o, real v, float) { __stcs(p + o, float(v)); }
  // pairs of values as stored: two consecutive ones at an even offset (one
  // 8-byte access) or two single ones; their values; the store of a pair
  using Raw = F2;
  __device__ static Raw raw2(const T* p) { return f2_of(__ldcs(reinterpret_cast<const float2*>(p))); }
  __device__ static Raw raw2g(const T* p) { return f2_of(__ldg(reinterpret_cast<const float2*>(p))); }
  __device__ static Raw raw11(const T* a, const T* b) { return F2(__ldg(a), __ldg(b)); }
  __device__ static Raw raw_of(T a, T b) { return F2(a, b); }
  __device__ static F2 value(Raw v, float) { return v; }
  __device__ static void st2_stream(T* p, F2 v, float) { __stcs(reinterpret_cast<float2*>(p), f2_in(v)); }
  // the same from shared memory, the rounded pair and its halves
  __device__ static Raw raw2s(const T* p) { return f2_of(*reinterpret_cast<const float2*>(p)); }
  __device__ static Raw raw11s(const T* p) { return F2(p[0], p[1]); }
  __device__ static Raw pack(F2 v, float) { return v; }
  __device__ static T half_of(Raw q, int k) { return k ? q.y : q.x; }
  __device__ static void st2_raw(T* p, Raw q) { __stcs(reinterpret_cast<float2*>(p), f2_in(q)); }
  // the values of one 16-byte load, as stored; one value
  static constexpr int kGroup = 4;
  __device__ static void group(const T* p, float* v) {
    const float4 q = __ldg(reinterpret_cast<const float4*>(p));
    v[0] = q.x; v[1] = q.y; v[2] = q.z; v[3] = q.w;
  }
  __device__ static float deviation(const T* p) { return __ldg(p); }
};
template <> struct Store<Fp16Dev> {
  using T = __half;
  template <typename real, typename I> __device__ static real ld(const T* p, I o, float ref) {
    return real(__half2float(__ldg(p + o)) + ref);
  }
  template <typename real, typename I> __device__ static real ld_last(const T* p, I o, float ref) {
    return real(__half2float(__ldcs(p + o)) + ref);
  }
  template <typename real, typename I> __device__ static void st(T* p, I o, real v, float ref) {
    p[o] = __float2half_rn(float(v) - ref);
  }
  template <typename real, typename I> __device__ static void st_stream(T* p, I o, real v, float ref) {
    __stcs(p + o, __float2half_rn(float(v) - ref));
  }
  // pairs of values as stored: two consecutive ones at an even offset (one
  // 4-byte access) or two single ones; their values; the store of a pair
  using Raw = __half2;
  __device__ static Raw raw2(const T* p) {
    const unsigned q = __ldcs(reinterpret_cast<const unsigned*>(p));
    return *reinterpret_cast<const __half2*>(&q);
  }
  __device__ static Raw raw2g(const T* p) {
    const unsigned q = __ldg(reinterpret_cast<const unsigned*>(p));
    return *reinterpret_cast<const __half2*>(&q);
  }
  __device__ static Raw raw11(const T* a, const T* b) { return __halves2half2(__ldg(a), __ldg(b)); }
  __device__ static Raw raw_of(T a, T b) { return __halves2half2(a, b); }
  __device__ static F2 value(Raw v, float ref) { return f2_of(__half22float2(v)) + F2(ref); }
  __device__ static void st2_stream(T* p, F2 v, float ref) {
    st2_raw(p, pack(v, ref));
  }
  // the same from shared memory (p odd for raw11s: the halves of two words), the
  // rounded pair and its halves
  __device__ static Raw raw2s(const T* p) { return *reinterpret_cast<const __half2*>(p); }
  __device__ static Raw raw11s(const T* p) {
    const unsigned a = *reinterpret_cast<const unsigned*>(p - 1), b = *reinterpret_cast<const unsigned*>(p + 1);
    const unsigned q = __byte_perm(a, b, 0x5432);
    return *reinterpret_cast<const __half2*>(&q);
  }
  __device__ static Raw pack(F2 v, float ref) { return __float22half2_rn(f2_in(v - F2(ref))); }
  __device__ static T half_of(Raw q, int k) { return k ? __high2half(q) : __low2half(q); }
  __device__ static void st2_raw(T* p, Raw q) {
    __stcs(reinterpret_cast<unsigned*>(p), *reinterpret_cast<const unsigned*>(&q));
  }
  // the deviations of one 16-byte load, without the reference; one deviation
  static constexpr int kGroup = 8;
  __device__ static void group(const T* p, float* v) {
    const uint4 q = __ldg(reinterpret_cast<const uint4*>(p));
    const unsigned w[4] = {q.x, q.y, q.z, q.w};
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const float2 f = __half22float2(*reinterpret_cast<const __half2*>(&w[k]));
      v[2 * k] = f.x;
      v[2 * k + 1] = f.y;
    }
  }
  __device__ static float deviation(const T* p) { return __half2float(__ldg(p)); }
};

// ---------------------------------------------------------------------------
// bounds-check builds (-DLBM_BOUNDS_CHECK): every population access of the
// step kernels must lie inside one of the handle's two population buffers;
// one outside is skipped (a load gives 0) and counted: every element of a pull and of
// a bulk copy with its side units, the elements of a vector load or store together.
// Other builds compile the check away.
// ---------------------------------------------------------------------------
#ifdef LBM_BOUNDS_CHECK
namespace {
__device__ unsigned long long g_oob;                 // accesses outside the buffers (this unit's kernels)
unsigned long long read_oob() {
  unsigned long long v = 0;
  cudaMemcpyFromSymbol(&v, g_oob, sizeof(v));
  return v;
}
struct OobReaderRegistration {
  OobReaderRegistration() { register_oob_reader(&read_oob); }
} g_oob_registration;
}  // namespace
#endif

// the n elements ptr[off .. off + n) are inside a population buffer of p (not counted)
template <typename T>
__device__ __forceinline__ bool pop_inside(const Params& p, const T* ptr, long long off, int n) {
#ifdef LBM_BOUNDS_CHECK
  const T* a = ptr + off;
  const long long len = 2LL * p.Q * p.plane;
  for (int k = 0; k < 2; ++k) {
    const T* lo = static_cast<const T*>(p.pop[k]);
    if (lo && a >= lo && a + n <= lo + len) return a + n <= lo + p.hide_lo || a >= lo + p.hide_hi;
  }
  return false;
#else
  return true;
#endif
}
// the same, an access outside counted
template <typename T>
__device__ __forceinline__ bool pop_ok(const Params& p, const T* ptr, long long off, int n = 1) {
#ifdef LBM_BOUNDS_CHECK
  if (pop_inside(p, ptr, off, n)) return true;
  atomicAdd(&g_oob, 1ULL);
  return false;
#else
  return true;
#endif
}

// one population value as stored, checked; 0 outside
template <typename T> __device__ __forceinline__ T pop_value(const Params& p, const T* a) {
  return pop_ok(p, a, 0) ? __ldg(a) : T(0.f);
}

// ---------------------------------------------------------------------------
// geometry helpers
// ---------------------------------------------------------------------------
__device__ __forceinline__ int wrap(int v, int n) { return v < 0 ? v + n : (v >= n ? v - n : v); }

__device__ __forceinline__ long long node_off(const Params& p, int xp, int y, int z) {
  return ((long long)z * p.Ny + y) * p.pitch + xp;
}

// padded x of interior coordinate x (+ shift), wrapped when x is periodic
__device__ __forceinline__ int xpad(const Params& p, int xp_shifted) {
  return p.periodic_x ? wrap(xp_shifted, p.Nx) : xp_shifted;
}

// x of the node whose density the Laplacian of the Korteweg force (Eq. FK)
// reads at interior coordinate gx: gx itself, or its mirror image across a
// wall face when gx is a ghost column of that face (the wall is a symmetry
// plane of the capillary terms)
__host__ __device__ __forceinline__ int wall_mirror(const Params& p, int gx) {
  if (gx < 0 && p.bc_lo == LBM_BC_WALL) return -1 - gx;
  if (gx >= p.Nx && p.bc_hi == LBM_BC_WALL) return 2 * p.Nx - 1 - gx;
  return gx;
}

// decode a linear index over [xlo, xhi) x Ny x Nz (padded x)
__device__ __forceinline__ bool decode(const Params& p, long long gid, int xlo, int xhi, int& xp, int& y, int& z) {
  const int nx = xhi - xlo;
  const long long n = (long long)nx * p.Ny * p.Nz;
  if (gid >= n) return false;
  xp = xlo + int(gid % nx);
  long long r = gid / nx;
  y = int(r % p.Ny);
  z = int(r / p.Ny);
  return true;
}

// Primitive state at interior coordinate (x, y, z) extended by the x-face
// rules: inflow faces give their prescribed state, outflow faces the nearest
// interior node, wall faces the nearest interior node's density with the
// wall's velocity and temperature, periodic wraps.  rho, u (D planes), T:
// interior FP64 fields.
template <int D>
__device__ inline void prim_ext(const Params& p, const double* rho, const double* u, const double* T,
                                int x, int y, int z, double& r, double* uu, double& t) {
  const long long N = (long long)p.Nx * p.Ny * p.Nz;
  const double* st = nullptr;
  const double* wall = nullptr;
  if (p.periodic_x) {
    x = wrap(x, p.Nx);
  } else if (x < 0) {
    if (p.bc_lo == LBM_BC_INFLOW) st = p.st_lo; else x = 0;
    if (p.bc_lo == LBM_BC_WALL) wall = p.st_lo;
  } else if (x >= p.Nx) {
    if (p.bc_hi == LBM_BC_INFLOW) st = p.st_hi; else x = p.Nx - 1;
    if (p.bc_hi == LBM_BC_WALL) wall = p.st_hi;
  }
  if (st) {
    r = st[0];
    for (int a = 0; a < D; ++a) uu[a] = st[1 + a];
    t = st[4];
    return;
  }
  const long long n = x + (long long)p.Nx * (y + (long long)p.Ny * z);
  r = rho[n];
  for (int a = 0; a < D; ++a) uu[a] = wall ? wall[1 + a] : u[a * N + n];
  t = wall ? wall[4] : T[n];
}

// ---------------------------------------------------------------------------
// index arithmetic: flattened node index -> (x, y, z) by
// multiplication (Granlund and Montgomery, "Division by invariant integers
// using multiplication", 1994: exact for n < 2^31)
// ---------------------------------------------------------------------------
struct FastDiv {
  unsigned d, m, s;
  __host__ __device__ FastDiv() : d(1), m(1), s(0) {}                     // by one
  __host__ explicit FastDiv(unsigned d_) : d(d_), s(0) {
    while ((1ull << s) < d) ++s;
    m = unsigned(((1ull << 32) * ((1ull << s) - d)) / d + 1);
  }
  __device__ __forceinline__ unsigned div(unsigned n) const { return (__umulhi(n, m) + n) >> s; }
};

// nodes (or groups of `quad` nodes along x) of the padded-x range [lo, hi) x Ny x Nz
struct NodeRange {
  int lo, quad;
  unsigned n;
  FastDiv nx, ny;
  __host__ NodeRange() : lo(0), quad(1), n(0) {}
  __host__ NodeRange(const Params& p, int lo_, int hi_, int quad_ = 1)
      : lo(lo_), quad(quad_), nx(unsigned((hi_ - lo_ + quad_ - 1) / quad_)), ny(unsigned(p.Ny)) {
    n = nx.d * unsigned(p.Ny) * unsigned(p.Nz);
  }
  __device__ __forceinline__ bool decode(unsigned gid, int& xp, int& y, int& z) const {
    if (gid >= n) return false;
    const unsigned r = nx.div(gid), q = ny.div(r);
    xp = lo + int(gid - r * nx.d) * quad;
    y = int(r - q * ny.d);
    z = int(q);
    return true;
  }
};

// x range (padded) of the moment region: radius r beyond the interior
__host__ __device__ inline void moment_range(const Params& p, int r, int& lo, int& hi) {
  if (p.periodic_x) { lo = 0; hi = p.Nx; }
  else { lo = p.G - r; hi = p.G + p.Nx + r; }
}

// in-plane element offsets of the 3^D source nodes of one node (x - c): row
// part per (c_y[, c_z]) and x part per c_x; a population's plane base is
// uniform, so a load costs one addition
template <int D> struct PullOffsets {
  unsigned x[3], r[D == 3 ? 9 : 3];
  __device__ __forceinline__ PullOffsets() {}
  __device__ __forceinline__ PullOffsets(const Params& p, int xp, int y, int z) {
    rows(p, y, z);
#pragma unroll
    for (int c = -1; c <= 1; ++c) x[c + 1] = unsigned(xpad(p, xp - c));
  }
  __device__ __forceinline__ void rows(const Params& p, int y, int z) {
    const unsigned pitch = unsigned(p.pitch), zs = pitch * unsigned(p.Ny);
#pragma unroll
    for (int cz = (D == 3 ? -1 : 0); cz <= (D == 3 ? 1 : 0); ++cz)
#pragma unroll
      for (int cy = -1; cy <= 1; ++cy)
        r[(D == 3 ? 3 * (cz + 1) : 0) + cy + 1] =
            unsigned(wrap(y - cy, p.Ny)) * pitch + (D == 3 ? unsigned(wrap(z - cz, p.Nz)) * zs : 0u);
  }
  // row offset of direction i's source
  __device__ __forceinline__ unsigned row(int i) const {
    using L = Lattice<D>;
    return r[D == 3 ? 3 * (L::c(i, D - 1) + 1) + L::c(i, 1) + 1 : L::c(i, 1) + 1];
  }
  __device__ __forceinline__ unsigned operator()(int i) const { return row(i) + x[Lattice<D>::c(i, 0) + 1]; }
};

// ---------------------------------------------------------------------------
// initialisation: pulled value at every node used by a step = equilibrium of
// the (extended) initial primitive state there (Fig. FlowChart, Initialize).
// Thread per source node x in [-G-1, Nx+G] (bounded) or [0, Nx) (periodic);
// writes A_i(x - c_i) = eq_i(x), which is what node x - c_i + c_i = x pulls.
// ---------------------------------------------------------------------------
// (Params as a grid constant: prim_ext takes the address of its inflow state,
// which would otherwise copy the whole parameter block to local memory)
template <int D, typename S>
__global__ void __launch_bounds__(128) k_init(const __grid_constant__ Params p, typename Store<S>::T* A,
                                              const double* rho, const double* u, const double* T) {
  using L = Lattice<D>;
  const int xlo = p.periodic_x ? 0 : -p.G - 1;
  const int xhi = p.periodic_x ? p.Nx : p.Nx + p.G + 1;
  int x, y, z;
  if (!decode(p, blockIdx.x * (long long)blockDim.x + threadIdx.x, xlo, xhi, x, y, z)) return;
  double r, uu[D], t;
  prim_ext<D>(p, rho, u, T, x, y, z, r, uu, t);
  Model<double> m = model_of<double>(p);
  const int NxP = p.Nx + 2 * p.G;
  auto put = [&](int i, int ii, double v) {
    int xs = x - L::c(i, 0) + p.G;
    if (p.periodic_x) xs = wrap(xs, p.Nx);
    else if (xs < 0 || xs >= NxP) return;
    const int ys = wrap(y - L::c(i, 1), p.Ny);
    const int zs = D == 3 ? wrap(z - L::c(i, 2), p.Nz) : z;
    const long long o = ii * p.plane + node_off(p, xs, ys, zs);
    if (pop_ok(p, A, o)) Store<S>::template st<double>(A, o, v, p.ref[ii]);
  };
  equilibria_of<D>(r, uu, eos_pressure(m, r, t) / r, eos_energy(m, r, t), [&](int i, double v) { put(i, i, v); },
                   [&](int i, double v) { put(i, L::Q + i, v); });
}

// The same for populations stored in FP32 or less, in packed double-float
// arithmetic: two nodes per thread, 32 apart, so that every store of a warp is
// a full line.  The FP64 form is bound by the FP64 pipe (425 instructions per
// node, 11.4 ms at 256^3 against 0.6 ms of memory traffic).  Its values, rounded to FP32,
// are these but for those that lie next to the middle between two FP32 numbers: 7 of 150
// million values over the states of the scenarios, off by at most 1.5e-6 ulp more than the
// half (relative L2 error of the stored populations the same to 12 digits); with densities
// up to 2.6 of the limit 3 and |u| up to 0.4 at random 2e-6 of the values, one by 1.1 ulp.
struct InitConsts {
  float a[2], b[2], R[2], cv[2];             // model constants as high and low parts
  __host__ explicit InitConsts(const Params& p) {
    auto split = [](double v, float* s) {
      s[0] = float(v);
      s[1] = float(v - double(s[0]));
    };
    split(p.a, a);
    split(p.b, b);
    split(p.R, R);
    split(p.cv, cv);
  }
};

template <int D, typename S>
__global__ void __launch_bounds__(128) k_init_df(const __grid_constant__ Params p, const InitConsts c,
                                                 const NodeRange range, typename Store<S>::T* A, const double* rho,
                                                 const double* u, const double* T) {
  using L = Lattice<D>;
  using ST = typename Store<S>::T;
  const unsigned gid = blockIdx.x * 256u + (threadIdx.x >> 5) * 64u + (threadIdx.x & 31u);
  int x[2], y[2], z[2];
  bool act[2];
#pragma unroll
  for (int k = 0; k < 2; ++k) act[k] = range.decode(gid + 32u * k, x[k], y[k], z[k]);
  if (!act[0]) return;
  if (!act[1]) { x[1] = x[0]; y[1] = y[0]; z[1] = z[0]; }
  double r[2], uu[2][D], t[2];
#pragma unroll
  for (int k = 0; k < 2; ++k) prim_ext<D>(p, rho, u, T, x[k], y[k], z[k], r[k], uu[k], t[k]);
  DF2 theta, e, ud[D];
  const DF2 rd = df_of(r[0], r[1]);
#pragma unroll
  for (int a = 0; a < D; ++a) ud[a] = df_of(uu[0][a], uu[1][a]);
  if (p.eos_kind == LBM_EOS_PR) {
    const Model<double> m = model_of<double>(p);
    theta = df_of(pr_pressure(m, r[0], t[0]) / r[0], pr_pressure(m, r[1], t[1]) / r[1]);
    e = df_of(pr_energy(m, r[0], t[0]), pr_energy(m, r[1], t[1]));
  } else {
    auto cst = [](const float* v) { return DF2(F2(v[0]), F2(v[1])); };
    const DF2 td = df_of(t[0], t[1]), ar = cst(c.a) * rd;
    theta = cst(c.R) * td * df_inverse(DF2(1.f) - cst(c.b) * rd) - ar;         // P / rho of Eq. Pvdw
    e = cst(c.cv) * td - ar;
  }
  // destinations: row offsets and x of both nodes (dropped past the ends of a bounded row)
  unsigned ro[2][D == 3 ? 9 : 3], xo[2][3];
  bool in[2][3];
#pragma unroll
  for (int k = 0; k < 2; ++k) {
    PullOffsets<D> po;
    po.rows(p, y[k], z[k]);
#pragma unroll
    for (int q = 0; q < (D == 3 ? 9 : 3); ++q) ro[k][q] = po.r[q];
#pragma unroll
    for (int cx = -1; cx <= 1; ++cx) {
      const int xs = p.periodic_x ? wrap(x[k] - cx, p.Nx) : x[k] - cx + p.G;
      in[k][cx + 1] = act[k] && (p.periodic_x || (xs >= 0 && xs < p.Nx + 2 * p.G));
      xo[k][cx + 1] = unsigned(xs);
    }
  }
  auto put = [&](int i, int ii, F2 v) {
    ST* Ai = A + (long long)ii * p.plane;
    const int q = D == 3 ? 3 * (L::c(i, D - 1) + 1) + L::c(i, 1) + 1 : L::c(i, 1) + 1, cx = L::c(i, 0) + 1;
    const auto w = Store<S>::pack(v, p.ref[ii]);
    const unsigned o0 = ro[0][q] + xo[0][cx], o1 = ro[1][q] + xo[1][cx];
    if (in[0][cx] && pop_ok(p, Ai, o0)) Ai[o0] = Store<S>::half_of(w, 0);
    if (in[1][cx] && pop_ok(p, Ai, o1)) Ai[o1] = Store<S>::half_of(w, 1);
  };
  equilibria_of<D>(rd, ud, theta, e, [&](int i, F2 v) { put(i, i, v); }, [&](int i, F2 v) { put(i, L::Q + i, v); });
}

// ---------------------------------------------------------------------------
// split step, pass 1: moments rho, j = sum c f, S = sum g (Eqs. def_h, def_u,
// def_E) of the pulled populations, on the interior plus 3 ghost layers.
// M planes: rho, j_0..j_{D-1}, S   (each p.plane elements, padded layout)
// Each component of j is (sum over c_a = +1) minus (sum over c_a = -1), the two
// summed in the same order: exactly zero for mirror-symmetric populations.
// One read of every population bounds it.
// ---------------------------------------------------------------------------
// FP64: one node per thread
template <int D>
__device__ __forceinline__ void moments_nodes(const Params& p, const NodeRange& range, const double* __restrict__ A, double* __restrict__ M, const unsigned block) {
  using L = Lattice<D>;
  int xp, y, z;
  if (!range.decode(block * blockDim.x + threadIdx.x, xp, y, z)) return;
  const PullOffsets<D> po(p, xp, y, z);
  auto pulled = [&](const int i, const int ii) {
    const double* Ai = A + (long long)ii * p.plane;
    return pop_ok(p, Ai, po(i)) ? __ldg(Ai + po(i)) : 0.0;
  };
  const unsigned o = po.r[D == 3 ? 4 : 1] + unsigned(xp);
  double rho = 0.0, S = 0.0, sp[D], sn[D];
#pragma unroll
  for (int a = 0; a < D; ++a) sp[a] = sn[a] = 0.0;
#pragma unroll
  for (int i = 0; i < L::Q; ++i) {
    const double v = pulled(i, i);
    rho += v;
#pragma unroll
    for (int a = 0; a < D; ++a) {
      if (L::c(i, a) == 1) sp[a] += v;
      if (L::c(i, a) == -1) sn[a] += v;
    }
  }
#pragma unroll
  for (int i = 0; i < L::Q; ++i) S += pulled(i, L::Q + i);
  M[o] = rho;
#pragma unroll
  for (int a = 0; a < D; ++a) M[(1 + a) * p.plane + o] = sp[a] - sn[a];
  M[(1 + D) * p.plane + o] = S;
}
template <int D>
__global__ void __launch_bounds__(256) k_moments(const __grid_constant__ Params p, const NodeRange range,
                                                 const double* __restrict__ A, double* __restrict__ M) {
  wait_previous_launch();
  moments_nodes<D>(p, range, A, M, blockIdx.x);
}

// FP32 arithmetic: the nodes of one 16-byte load (4 FP32, 8 FP16-deviation
// values) per thread, packed sums; a direction with c_x != 0 takes one scalar
// load for the node pulled from outside the group.  FP16-deviation: the stored
// deviations are summed and the reference populations' sum added once (in j the
// references of mirrored directions cancel).  RAGGED: a row's last group holds
// fewer nodes, its last one pulls across the seam.  With four nodes (8-byte
// loads) FP16-deviation issued as many loads as FP32 for half the bytes: 584 us
// at 256^3, against FP32's 560 (7 TB/s); with whole groups 314 and 550 us.
template <int D, typename S, bool RAGGED>
__device__ __forceinline__ void moments_groups(const Params& p, const NodeRange& range, const typename Store<S>::T* __restrict__ A,
                                              float* __restrict__ M, const unsigned block) {
  using L = Lattice<D>;
  using ST = typename Store<S>::T;
  constexpr int N = Store<S>::kGroup, H = N / 2, T3 = L::Q / 3;
  int xp, y, z;
  if (!range.decode(block * blockDim.x + threadIdx.x, xp, y, z)) return;
  PullOffsets<D> po;
  po.rows(p, y, z);
  // the node that pulls from right of the group, and the sources left and right
  // (kept inside the row where the pulled value is not used)
  const int last = RAGGED && p.periodic_x ? min(N, p.Nx - xp) - 1 : N - 1;
  const unsigned xl = unsigned(p.periodic_x ? wrap(xp - 1, p.Nx) : max(xp - 1, 0));
  const unsigned xr = unsigned(p.periodic_x ? wrap(xp + last + 1, p.Nx) : min(xp + N, p.pitch - 1));
  const unsigned o = po.r[D == 3 ? 4 : 1] + unsigned(xp);
  auto put = [&](const int k, const F2* v) {
    float* dst = M + (long long)k * p.plane + o;
#pragma unroll
    for (int q = 0; q < H; q += 2) *reinterpret_cast<float4*>(dst + 2 * q) = make_float4(v[q].x, v[q].y, v[q + 1].x, v[q + 1].y);
  };
  // the group's values of direction i, as pulled
  auto pulled = [&](const int i, const int ii, F2* v) {
    const int cx = L::c(i, 0);
    const ST* Ai = A + (long long)ii * p.plane + po.row(i);
    float w[N], e = 0.f;
    if (pop_ok(p, Ai, xp, N)) Store<S>::group(Ai + xp, w);
    else
#pragma unroll
      for (int j = 0; j < N; ++j) w[j] = 0.f;
    if (cx != 0 && pop_ok(p, Ai, cx > 0 ? xl : xr)) e = Store<S>::deviation(Ai + (cx > 0 ? xl : xr));
    float q[N];
#pragma unroll
    for (int j = 0; j < N; ++j) {
      if (cx > 0) q[j] = j == 0 ? e : w[j - (j > 0)];
      else if (cx < 0) q[j] = j == N - 1 ? e : (RAGGED && j == last ? e : w[j + (j < N - 1)]);
      else q[j] = w[j];
    }
#pragma unroll
    for (int j = 0; j < H; ++j) v[j] = F2(q[2 * j], q[2 * j + 1]);
  };
  F2 rho[H], jx[H], sp[2][H], sn[2][H], b[H], v[H];
#pragma unroll
  for (int j = 0; j < H; ++j) {
    rho[j] = jx[j] = F2(0.f);
#pragma unroll
    for (int a = 0; a < 2; ++a) sp[a][j] = sn[a][j] = F2(0.f);
  }
#pragma unroll
  for (int c = 0; c < 3; ++c) {                              // the directions of one c_x
#pragma unroll
    for (int j = 0; j < H; ++j) b[j] = F2(0.f);
#pragma unroll
    for (int k = 0; k < T3; ++k) {
      const int i = c * T3 + k;
      pulled(i, i, v);
#pragma unroll
      for (int j = 0; j < H; ++j) {
        b[j] += v[j];
#pragma unroll
        for (int a = 1; a < D; ++a) {
          if (L::c(i, a) == 1) sp[a - 1][j] += v[j];
          if (L::c(i, a) == -1) sn[a - 1][j] += v[j];
        }
      }
    }
#pragma unroll
    for (int j = 0; j < H; ++j) {
      rho[j] += b[j];
      if (c == 0) jx[j] = b[j];                              // c_x = -1
      if (c == 2) jx[j] = b[j] - jx[j];
    }
  }
#pragma unroll
  for (int j = 0; j < H; ++j) {
    rho[j] += F2(p.refsum[0]);
#pragma unroll
    for (int a = 0; a < 2; ++a) sp[a][j] = sp[a][j] - sn[a][j];
  }
  put(0, rho);
  put(1, jx);
#pragma unroll
  for (int a = 1; a < D; ++a) put(1 + a, sp[a - 1]);
#pragma unroll
  for (int j = 0; j < H; ++j) rho[j] = F2(0.f);
#pragma unroll
  for (int i = 0; i < L::Q; ++i) {
    pulled(i, L::Q + i, v);
#pragma unroll
    for (int j = 0; j < H; ++j) rho[j] += v[j];
  }
#pragma unroll
  for (int j = 0; j < H; ++j) rho[j] += F2(p.refsum[1]);
  put(1 + D, rho);
}
template <int D, typename S, bool RAGGED>
__global__ void __launch_bounds__(128) k_moments_row(const __grid_constant__ Params p, const NodeRange range,
                                                     const typename Store<S>::T* __restrict__ A,
                                                     float* __restrict__ M) {
  wait_previous_launch();
  moments_groups<D, S, RAGGED>(p, range, A, M, blockIdx.x);
}

// neighbour offset along axis a by s (wrapping periodic axes)
__device__ __forceinline__ unsigned nb_off(const Params& p, int xp, int y, int z, int a, int s) {
  if (a == 0) xp = xpad(p, xp + s);
  else if (a == 1) y = wrap(y + s, p.Ny);
  else z = wrap(z + s, p.Nz);
  return unsigned(node_off(p, xp, y, z));
}

// compact Laplacian of rho at (xp, y, z); ghost columns of a wall face read
// their mirror image (wall_mirror)
template <int D, typename real>
__device__ __forceinline__ real lap_rho(const Params& p, const real* rho, int xp, int y, int z) {
  const int xc = wall_mirror(p, xp - p.G) + p.G;
  const real c = rho[node_off(p, xc, y, z)];
  const int xr = wall_mirror(p, xpad(p, xp + 1) - p.G) + p.G, xl = wall_mirror(p, xpad(p, xp - 1) - p.G) + p.G;
  real l = rho[node_off(p, xr, y, z)] - real(2) * c + rho[node_off(p, xl, y, z)];
#pragma unroll
  for (int a = 1; a < D; ++a) l += rho[nb_off(p, xc, y, z, a, 1)] - real(2) * c + rho[nb_off(p, xc, y, z, a, -1)];
  return l;
}

__device__ __forceinline__ void shift(const Params& p, int& xp, int& y, int& z, int a, int s) {
  if (a == 0) xp = xpad(p, xp + s);
  else if (a == 1) y = wrap(y + s, p.Ny);
  else z = wrap(z + s, p.Nz);
}

// What a closure hands on to the collision besides T: nothing (h, Lambda and e of a van
// der Waals node follow from rho, u and T); P and c_s^2 with h and Lambda (kExtra
// closures); or e (kEnergy closures: T inverted in FP64, where T rounded to FP32 would
// not give e back).
enum Handed { kHandNothing, kHandState, kHandEnergy };
template <class CL> constexpr Handed handed() {
  return CL::kExtra > 0 ? kHandState : (CL::kEnergy ? kHandEnergy : kHandNothing);
}

// Planes of the primitive fields W (split step): u_a, T, F_a; h and Lam_a, unless
// the collision takes them from rho, u and T (derives_fields), where e may stand in
// h's place; with a closure that hands them on, P and c_s^2.
template <int D> struct WPlanes {
  static constexpr int U = 0, T = D, H = D + 1, E = H, LAM = D + 2, F = 2 * D + 2, P = 3 * D + 2, CS2 = 3 * D + 3;
};

// h and Lambda of a van der Waals node are functions of rho, u_a and T alone: in FP32
// arithmetic the collision, bound by memory, evaluates them at the node and its
// neighbours instead of reading four more planes that the pass before wrote
// (256^3: 1917 -> 1838 us per step in FP32, 1382 -> 1263 with FP16 deviations).  In
// FP64, bound by the FP64 units, they stay planes; with P and c_s^2 handed on they
// have no such form.
template <typename real, Handed HD> constexpr bool derives_fields() { return sizeof(real) == 4 && HD != kHandState; }

// The Korteweg force of a 3-D node is the difference of the density's Laplacian
// across it: FP32 steps hand the Laplacian on, one plane (in F's place) for three
// (256^3: 1838 -> 1807 us per step in FP32, 1260 -> 1240 with FP16 deviations).
template <int D, typename real> constexpr bool hands_laplacian() { return D == 3 && sizeof(real) == 4; }

// e of a node whose closure hands on h = e + P / rho and P: the same quotient must be
// taken off that prims_node put on.  Both round it exactly (Divider); with two different
// approximations of it the total energy of a Peng-Robinson box drifted by -9.0e-9 (rho
// 0.45) to +3.1e-9 (rho 0.4) of itself per step, now by at most 0.1e-9.
template <typename V> __device__ __forceinline__ V handed_energy(V h, V P, V rho) { return h - Divider<V>(rho)(P); }

// Primitive fields of one node from its moments and the Korteweg force F:
// u, E, the closure's (T, P, c_s^2, e), then h and Lambda, stored at offset o.
// Warp-collective closures need every lane of the warp (act: a real node).
template <int D, typename real, class CL>
__device__ __forceinline__ void prims_node(const Params& p, const Model<real>& m, const CL& closure, bool act,
                                           real rho, const real* j, real S, const real* F, real lap,
                                           real* __restrict__ W, unsigned o) {
  using WP = WPlanes<D>;
  real u[D], uF = real(0), u2 = real(0), E = real(0);
#pragma unroll
  for (int a = 0; a < D; ++a) u[a] = real(0);
  const Divider<real> over_rho(rho);
  if (act) {
#pragma unroll
    for (int a = 0; a < D; ++a) {
      u[a] = over_rho(mad(real(0.5), F[a], j[a]));                                      // Eq. def_u
      uF = mad(u[a], F[a], uF);
      u2 = mad(u[a], u[a], u2);
    }
    E = over_rho(mad(real(0.5), uF, S));                                                // Eq. def_E
  }
  real T = real(0), P = real(1), cs2 = real(0), e = real(0);
  if constexpr (CL::kWarp) closure(m, rho, E, u2, act, T, P, cs2, e);
  else if (act) closure(m, rho, E, u2, act, T, P, cs2, e);
  if (!act) return;
  constexpr bool kPlanes = !CL::kOutput && !derives_fields<real, handed<CL>()>();     // h and Lambda
  constexpr bool kLap = !CL::kOutput && hands_laplacian<D, real>();
  const real theta = over_rho(P);                                                       // rounded as handed_energy's
  auto put = [&](const int k, const real v) { W[(long long)k * p.plane + o] = v; };
#pragma unroll
  for (int a = 0; a < D; ++a) {
    put(WP::U + a, u[a]);
    if constexpr (kPlanes) put(WP::LAM + a, rho * u[a] * u[a] * u[a] + real(3) * rho * u[a] * (theta - real(1.0 / 3.0)));
    if constexpr (!kLap) put(WP::F + a, F[a]);
  }
  if constexpr (kLap) put(WP::F, lap);
  put(WP::T, T);
  if constexpr (kPlanes) put(WP::H, e + theta);                                         // Eq. enthalpy
  if constexpr (!CL::kOutput && handed<CL>() == kHandEnergy) put(WP::E, e);
  if constexpr (CL::kExtra > 0) {
    put(WP::P, P);
    put(WP::CS2, cs2);
  }
}

// ---------------------------------------------------------------------------
// split step, pass 2: Korteweg force and primitive fields on interior + 1
// ghost layer (2-D form: every value of the stencil read from memory).
// ---------------------------------------------------------------------------
template <int D, typename real, class CL>
__global__ void __launch_bounds__(256) k_prims(const __grid_constant__ Params p, const NodeRange range,
                                               const real* __restrict__ M, real* __restrict__ W) {
  wait_previous_launch();
  extern __shared__ __align__(128) unsigned char smem_raw[];
  CL closure;
  closure.load(p, smem_raw);
  if constexpr (CL::kSmem > 0) __syncthreads();
  int xp = 0, y = 0, z = 0;
  const bool act = range.decode(blockIdx.x * blockDim.x + threadIdx.x, xp, y, z);
  if (!CL::kWarp && !act) return;
  const Model<real> m = model_of<real>(p);
  real rho = real(1), j[D], F[D], S = real(0);
#pragma unroll
  for (int a = 0; a < D; ++a) j[a] = F[a] = real(0);
  const unsigned o = unsigned(node_off(p, xp, y, z));
  if (act) {
    rho = M[o];
    S = M[(1 + D) * p.plane + o];
#pragma unroll
    for (int a = 0; a < D; ++a) {
      int x1 = xp, y1 = y, z1 = z, x2 = xp, y2 = y, z2 = z;
      shift(p, x1, y1, z1, a, 1);
      shift(p, x2, y2, z2, a, -1);
      F[a] = m.kappa * rho * real(0.5) * (lap_rho<D, real>(p, M, x1, y1, z1) - lap_rho<D, real>(p, M, x2, y2, z2));  // Eq. FK
      j[a] = M[(1 + a) * p.plane + o];
    }
  }
  prims_node<D, real, CL>(p, m, closure, act, rho, j, S, F, real(0), W, o);
}

// ---------------------------------------------------------------------------
// split step, pass 2 in 3-D: a block of 32 x 8 threads marches z over a column
// of nodes with the density of three planes (radius 2 in the plane) and its
// Laplacian of three planes (radius 1) in shared memory: rho, j and S are read
// once, the Laplacian once computed per node instead of six times from 25
// loads.  The next plane's density and this plane's j, S are loaded before
// they are needed; two barriers per plane.  256^3 FP32: 711 us with every value of
// the stencil read from memory, 217 us in this form, 155 us (5.1 TB/s) since it hands
// on seven planes fewer.
// ---------------------------------------------------------------------------
constexpr int kPrimX = 32, kPrimY = 8;
template <typename real, class CL> struct PrimsSmem {
  real rho[3][(kPrimY + 4) * (kPrimX + 4)];
  real lap[3][(kPrimY + 2) * (kPrimX + 2)];
};
template <typename real, class CL, int MINB>
__device__ __forceinline__ void prims_column(const Params& p, int lo, int hi, int ncolx, int ncoly, int nseg,
                                             const real* __restrict__ M, real* __restrict__ W, const unsigned block) {
  constexpr int NT = kPrimX * kPrimY, BX2 = kPrimX + 4, BX1 = kPrimX + 2;
  constexpr int N2 = BX2 * (kPrimY + 4), N1 = BX1 * (kPrimY + 2), K2 = (N2 + NT - 1) / NT, K1 = (N1 + NT - 1) / NT;
  __shared__ PrimsSmem<real, CL> sm;
  extern __shared__ __align__(128) unsigned char smem_raw[];
  CL closure;
  closure.load(p, smem_raw);
  const Model<real> m = model_of<real>(p);
  const int tid = threadIdx.x, lx = tid % kPrimX, ly = tid / kPrimX;
  int b = block;
  const int x0 = lo + (b % ncolx) * kPrimX;
  b /= ncolx;
  const int y0 = (b % ncoly) * kPrimY, seg = b / ncoly;
  const int mb = int((long long)p.Nz * seg / nseg), me = int((long long)p.Nz * (seg + 1) / nseg);
  const unsigned zs = unsigned(p.Ny) * unsigned(p.pitch);
  // in-plane offsets of the density box positions of this thread (periodic
  // axes wrapped; on bounded x the mirror image across a wall, kept inside the
  // row where the value is not used)
  unsigned o2[K2];
#pragma unroll
  for (int k = 0; k < K2; ++k) {
    const int q = min(tid + k * NT, N2 - 1), bx = q % BX2, by = q / BX2;
    int x = x0 + bx - 2, y = y0 + by - 2;
    y %= p.Ny;
    y += y < 0 ? p.Ny : 0;
    if (p.periodic_x) {
      x %= p.Nx;
      x += x < 0 ? p.Nx : 0;
    } else {
      x = min(max(wall_mirror(p, x - p.G) + p.G, 0), p.pitch - 1);
    }
    o2[k] = unsigned(y) * unsigned(p.pitch) + unsigned(x);
  }
  const int xp = x0 + lx, y = y0 + ly;
  const bool node = xp < hi && y < p.Ny;
  const real* Mn = M + (node ? unsigned(y) * unsigned(p.pitch) + unsigned(xp) : 0u);
  real* Wn = W + (Mn - M);
  // box position of this thread's Laplacian nodes
  int c1[K1];
#pragma unroll
  for (int k = 0; k < K1; ++k) c1[k] = ((tid + k * NT) / BX1 + 1) * BX2 + (tid + k * NT) % BX1 + 1;
  const unsigned ztop = zs * unsigned(p.Nz);
  auto first = [&](int z) {                       // offset of plane z, any z
    z %= p.Nz;
    return unsigned(z < 0 ? z + p.Nz : z) * zs;
  };
  auto next = [&](unsigned zo) { return zo + zs == ztop ? 0u : zo + zs; };
  unsigned zl = first(mb - 2), zo = first(mb);    // plane to load next, plane of the next output
  real nxt[K2];
#pragma unroll
  for (int k = 0; k < K2; ++k) nxt[k] = __ldg(M + zl + o2[k]);
  real *r0 = sm.rho[0], *r1 = sm.rho[2], *r2 = sm.rho[1];      // density of planes pl, pl - 1, pl - 2
  real *l0 = sm.lap[0], *l1 = sm.lap[2], *l2 = sm.lap[1];      // Laplacian of planes pl (= pl - 3), pl - 1, pl - 2
  for (int pl = mb - 2; pl <= me + 1; ++pl) {
#pragma unroll
    for (int k = 0; k < K2; ++k)
      if (tid + k * NT < N2) r0[tid + k * NT] = nxt[k];
    if (pl < me + 1) {
      zl = next(zl);
#pragma unroll
      for (int k = 0; k < K2; ++k) nxt[k] = __ldg(M + zl + o2[k]);
    }
    const bool out = pl >= mb + 2, act = out && node;          // this iteration's node is on plane pl - 2
    real rho = real(1), S = real(0), j[3] = {real(0), real(0), real(0)};
    if (act) {
      rho = __ldg(Mn + zo);
#pragma unroll
      for (int a = 0; a < 3; ++a) j[a] = __ldg(Mn + (1 + a) * p.plane + zo);
      S = __ldg(Mn + 4 * p.plane + zo);
    }
    __syncthreads();
    // Laplacian of plane pl - 1 on radius 1
    if (pl >= mb) {
#pragma unroll
      for (int k = 0; k < K1; ++k) {
        if (tid + k * NT < N1) {
          const int c = c1[k];
          const real c2 = real(2) * r1[c];
          l1[tid + k * NT] = (r1[c + 1] + r1[c - 1] - c2) + (r0[c] + r2[c] - c2) + (r1[c + BX2] + r1[c - BX2] - c2);
        }
      }
    }
    __syncthreads();
    if (out) {
      const int c = (ly + 1) * BX1 + lx + 1;
      const real kr = m.kappa * rho * real(0.5);
      const real F[3] = {kr * (l2[c + 1] - l2[c - 1]), kr * (l2[c + BX1] - l2[c - BX1]), kr * (l1[c] - l0[c])};   // Eq. FK
      prims_node<3, real, CL>(p, m, closure, act, rho, j, S, F, l2[c], Wn, zo);
      zo = next(zo);
    }
    real* t = r2;
    r2 = r1;
    r1 = r0;
    r0 = t;
    t = l2;
    l2 = l1;
    l1 = l0;
    l0 = t;
  }
}
template <typename real, class CL, int MINB>
__global__ void __launch_bounds__(kPrimX * kPrimY, MINB) k_prims3(const __grid_constant__ Params p, int lo, int hi, int ncolx,
                                                           int ncoly, int nseg, const real* __restrict__ M,
                                                           real* __restrict__ W) {
  wait_previous_launch();
  prims_column<real, CL, MINB>(p, lo, hi, ncolx, ncoly, nseg, M, W, blockIdx.x);
}

// ---------------------------------------------------------------------------
// split step, pass 3: derivatives and collision of every interior node (Eqs.
// fLBGK, gLBGK), written to dst at the node (pull scheme).  HD: what the closure
// handed on.
// ---------------------------------------------------------------------------
template <int D, typename S, typename real, Handed HD, int NTB, int MINB>
__device__ __forceinline__ void collide_nodes(const Params& p, const NodeRange& range, const typename Store<S>::T* __restrict__ A,
                                              typename Store<S>::T* __restrict__ B, const real* __restrict__ M,
                                              const real* __restrict__ W, unsigned* err, const unsigned block) {
  using L = Lattice<D>;
  using ST = typename Store<S>::T;
  using WP = WPlanes<D>;
  int xp, y, z;
  if (!range.decode(block * NTB + threadIdx.x, xp, y, z)) return;
  const PullOffsets<D> po(p, xp, y, z);
  const unsigned o = po.r[D == 3 ? 4 : 1] + unsigned(xp);
  real v[L::Q];
  // f populations first: in flight while the fields are read
#pragma unroll
  for (int i = 0; i < L::Q; ++i) {
    const ST* Ai = A + (long long)i * p.plane;
    v[i] = pop_ok(p, Ai, po(i)) ? Store<S>::template ld_last<real>(Ai, po(i), p.ref[i]) : real(0);
  }
  const Model<real> m = model_of<real>(p);
  auto w = [&](const int k, const unsigned at) { return __ldg(W + (long long)k * p.plane + at); };
  NodeState<D, real> s;
  s.rho = __ldg(M + o);
  s.T = w(WP::T, o);
  if constexpr (HD == kHandState) {
    s.P = w(WP::P, o);
    s.cs2 = w(WP::CS2, o);
    s.e = handed_energy(w(WP::H, o), s.P, s.rho);
  } else {
    s.P = vdw_pressure(m, s.rho, s.T);
    s.cs2 = vdw_cs2(m, s.rho, s.T);
    s.e = vdw_energy(m, s.rho, s.T);
  }
  s.sc = p.sc_on != 0;
  s.mu_num = s.eta_num = s.k_num = real(0);
  if (s.sc) {
    const real* V = static_cast<const real*>(p.sc_visc);
    s.mu_num = V[o];
    s.eta_num = V[p.plane + o];
    s.k_num = V[2 * p.plane + o];
  }
  s.div_u = 0;
#pragma unroll
  for (int a = 0; a < D; ++a) {
    s.u[a] = w(WP::U + a, o);
    s.F[a] = w(WP::F + a, o);
    const unsigned op = nb_off(p, xp, y, z, a, 1), om = nb_off(p, xp, y, z, a, -1);
    s.div_u += real(0.5) * (w(WP::U + a, op) - w(WP::U + a, om));
    s.gradT[a] = real(0.5) * (w(WP::T, op) - w(WP::T, om));
    s.gradh[a] = real(0.5) * (w(WP::H, op) - w(WP::H, om));
    const real lc = w(WP::LAM + a, o);
    const real back = lc - w(WP::LAM + a, om);
    const real fwd = w(WP::LAM + a, op) - lc;
    s.dLam[a] = upwind(s.u[a], back, fwd);
  }
  Attractors<D, real> at;
  at.setup(m, s);
  if (at.flags) atomicOr(err, at.flags);
  // f pass then g pass: one population set in flight at a time
  auto put = [&](const int i, const real x) {
    ST* Bi = B + (long long)i * p.plane;
    if (pop_ok(p, Bi, o)) Store<S>::template st_stream<real>(Bi, o, x, p.ref[i]);
  };
  FactoredRelax<D, real>::f_pass(at, [&](int i) { return v[i]; }, put);
#pragma unroll
  for (int i = 0; i < L::Q; ++i) {
    const ST* Ai = A + (long long)(L::Q + i) * p.plane;
    v[i] = pop_ok(p, Ai, po(i)) ? Store<S>::template ld_last<real>(Ai, po(i), p.ref[L::Q + i]) : real(0);
  }
  FactoredRelax<D, real>::g_pass(at, [&](int i) { return v[i]; }, [&](int i, real x) { put(L::Q + i, x); });
}
template <int D, typename S, typename real, Handed HD, int NTB, int MINB>
__global__ void __launch_bounds__(NTB, MINB)
k_collide(const __grid_constant__ Params p, const NodeRange range, const typename Store<S>::T* __restrict__ A,
          typename Store<S>::T* __restrict__ B, const real* __restrict__ M, const real* __restrict__ W,
          unsigned* err) {
  wait_previous_launch();
  collide_nodes<D, S, real, HD, NTB, MINB>(p, range, A, B, M, W, err, blockIdx.x);
}

// ---------------------------------------------------------------------------
// split step, pass 3 in FP32 arithmetic: two neighbouring nodes per thread
// (x = lo + 2k and the node right of it), one register pair per value, so that
// the collision's sums and products, the addresses and the stores cost one
// instruction for both.  Offsets are 32-bit byte offsets onto a plane base that
// is the same for every thread (a plane of a population is below 2^32 bytes:
// at most 2^32 / 18 elements of up to 8 bytes).
// Both population sets are requested before the fields are read: with 8 warps
// per multiprocessor (255 registers) the loads of one set alone leave the
// memory idle during the arithmetic.
// ODD: Nx odd; past the last node of a row the pair's second node is computed
// from in-row values and not stored.
// ---------------------------------------------------------------------------
template <typename T> __device__ __forceinline__ const T* at_bytes(const T* base, unsigned off) {
  return reinterpret_cast<const T*>(reinterpret_cast<const char*>(base) + off);
}
template <typename T> __device__ __forceinline__ T* at_bytes(T* base, unsigned off) {
  return reinterpret_cast<T*>(reinterpret_cast<char*>(base) + off);
}

template <int D, typename S, Handed HD, bool ODD, int NTB, int MINB>
__device__ __forceinline__ void collide_pairs(const Params& p, const NodeRange& range, const typename Store<S>::T* __restrict__ A,
                                              typename Store<S>::T* __restrict__ B, const float* __restrict__ M,
                                              const float* __restrict__ W, unsigned* err, const unsigned block) {
  using L = Lattice<D>;
  using ST = typename Store<S>::T;
  using WP = WPlanes<D>;
  constexpr unsigned ES = sizeof(ST);
  int xp, y, z;
  if (!range.decode(block * NTB + threadIdx.x, xp, y, z)) return;
  PullOffsets<D> po;                                         // rows in elements, then in bytes
  po.rows(p, y, z);
  const unsigned x = unsigned(xp), xm = unsigned(xpad(p, xp - 1)), x1 = unsigned(xpad(p, xp + 1)),
                 x2 = unsigned(xpad(p, xp + 2)), r0 = po.r[D == 3 ? 4 : 1], o = r0 + x;
  // rows of the neighbours along y and z
  unsigned nbp[D], nbm[D];
  nbp[0] = nbm[0] = 0;
  nbp[1] = po.r[(D == 3 ? 3 : 0) + 0] + x;                   // source of c_y = -1: y + 1
  nbm[1] = po.r[(D == 3 ? 3 : 0) + 2] + x;
  if constexpr (D == 3) {
    nbp[D - 1] = po.r[1] + x;
    nbm[D - 1] = po.r[7] + x;
  }
#pragma unroll
  for (int k = 0; k < (D == 3 ? 9 : 3); ++k) po.r[k] *= ES;
  const unsigned bx = x * ES, bm = xm * ES, b1 = x1 * ES, b2 = x2 * ES, bo = o * ES;
  const bool two = !ODD || xp + 1 < p.G + p.Nx;              // the second node is a node of the box
  auto pulled = [&](const int i, const int ii) {
    const ST* Ai = A + (long long)ii * p.plane;
    const int cx = L::c(i, 0);
    const unsigned r = po.row(i);
    const ST *a = at_bytes(Ai, r + (cx > 0 ? bm : (cx < 0 ? b1 : bx))), *b = cx == 0 ? a + 1 : at_bytes(Ai, r + (cx > 0 ? bx : b2));
#ifdef LBM_BOUNDS_CHECK
    return Store<S>::raw_of(pop_value(p, a), pop_value(p, b));
#endif
    return cx == 0 ? Store<S>::raw2(a) : Store<S>::raw11(a, b);
  };
  typename Store<S>::Raw v[2 * L::Q];
#pragma unroll
  for (int i = 0; i < L::Q; ++i) v[i] = pulled(i, i);
  const Model<float> m = model_of<float>(p);
  auto w1 = [&](const int k, const unsigned at) { return __ldg(at_bytes(W + (long long)k * p.plane, 4 * at)); };
  auto w2 = [&](const int k, const unsigned at) {
    return f2_of(__ldg(reinterpret_cast<const float2*>(at_bytes(W + (long long)k * p.plane, 4 * at))));
  };
  NodeState<D, F2> s;
  s.rho = f2_of(__ldg(reinterpret_cast<const float2*>(at_bytes(M, 4 * o))));
  s.T = w2(WP::T, o);
  constexpr bool DER = derives_fields<float, HD>(), LAP = hands_laplacian<D, float>();
  const F2 kr = F2(m.kappa) * s.rho * F2(0.5f);
  F2 h, theta, lap;
  if constexpr (LAP) lap = w2(WP::F, o);
  constexpr bool EN = HD == kHandEnergy;
  // h and theta = P / rho of a node pair from rho and T, and e where it is handed on
  auto enthalpy = [&](const F2 rho, const F2 T, const F2 e, F2& th) {
    const F2 hd = vdw_enthalpy(m, rho, T, th);
    return EN ? e + th : hd;
  };
  F2 e0(0.f), e1(0.f);
  if constexpr (EN) e0 = w2(WP::E, o);
  if constexpr (DER) h = enthalpy(s.rho, s.T, e0, theta);
  else h = w2(WP::H, o);
  s.sc = p.sc_on != 0;
  s.mu_num = s.eta_num = s.k_num = F2(0.f);
  if (s.sc) {
    const float* V = static_cast<const float*>(p.sc_visc);
    auto sc2 = [&](const int k) { return f2_of(__ldg(reinterpret_cast<const float2*>(V + k * p.plane + o))); };
    s.mu_num = sc2(0);
    s.eta_num = sc2(1);
    s.k_num = sc2(2);
  }
  s.div_u = F2(0.f);
#pragma unroll
  for (int a = 0; a < D; ++a) {
    s.u[a] = w2(WP::U + a, o);
    if constexpr (!LAP) s.F[a] = w2(WP::F + a, o);
    F2 lc, up, um, Tp, Tm, hp, hm, lp, lm;
    if constexpr (DER) lc = lambda_of(s.rho, s.u[a], theta);
    else lc = w2(WP::LAM + a, o);
    if (a == 0) {
      // neighbours of the pair are x - 1, the pair itself and x + 2; the node
      // right of a lone last node is read through its wrapped offset (into the
      // pair's second half)
      const bool lone = ODD && !two;
      const unsigned out2 = r0 + (lone ? x1 : x2), outm = r0 + xm;
      const F2 uo = F2(w1(WP::U, outm), w1(WP::U, out2)), To = F2(w1(WP::T, outm), w1(WP::T, out2));
      F2 ho, lo;
      if constexpr (DER) {
        const F2 ro = F2(__ldg(at_bytes(M, 4 * outm)), __ldg(at_bytes(M, 4 * out2)));
        F2 tho;
        if constexpr (EN) e1 = F2(w1(WP::E, outm), w1(WP::E, out2));
        ho = enthalpy(ro, To, e1, tho);
        lo = lambda_of(ro, uo, tho);
      } else {
        ho = F2(w1(WP::H, outm), w1(WP::H, out2));
        lo = F2(w1(WP::LAM, outm), w1(WP::LAM, out2));
      }
      if constexpr (LAP) {
        const F2 po2 = F2(w1(WP::F, outm), w1(WP::F, out2));
        s.F[0] = kr * (F2(lone ? po2.y : lap.y, po2.y) - F2(po2.x, lap.x));                  // Eq. FK
      }
      up = F2(lone ? uo.y : s.u[0].y, uo.y);
      um = F2(uo.x, s.u[0].x);
      Tp = F2(lone ? To.y : s.T.y, To.y);
      Tm = F2(To.x, s.T.x);
      hp = F2(lone ? ho.y : h.y, ho.y);
      hm = F2(ho.x, h.x);
      lp = F2(lone ? lo.y : lc.y, lo.y);
      lm = F2(lo.x, lc.x);
    } else {
      if constexpr (LAP) s.F[a] = kr * (w2(WP::F, nbp[a]) - w2(WP::F, nbm[a]));
      up = w2(WP::U + a, nbp[a]);
      um = w2(WP::U + a, nbm[a]);
      Tp = w2(WP::T, nbp[a]);
      Tm = w2(WP::T, nbm[a]);
      if constexpr (DER) {
        const F2 rp = f2_of(__ldg(reinterpret_cast<const float2*>(at_bytes(M, 4 * nbp[a])))),
                 rm = f2_of(__ldg(reinterpret_cast<const float2*>(at_bytes(M, 4 * nbm[a]))));
        F2 th;
        if constexpr (EN) e1 = w2(WP::E, nbp[a]);
        hp = enthalpy(rp, Tp, e1, th);
        lp = lambda_of(rp, up, th);
        if constexpr (EN) e1 = w2(WP::E, nbm[a]);
        hm = enthalpy(rm, Tm, e1, th);
        lm = lambda_of(rm, um, th);
      } else {
        hp = w2(WP::H, nbp[a]);
        hm = w2(WP::H, nbm[a]);
        lp = w2(WP::LAM + a, nbp[a]);
        lm = w2(WP::LAM + a, nbm[a]);
      }
    }
    s.div_u = mad(F2(0.5f), up - um, s.div_u);
    s.gradT[a] = F2(0.5f) * (Tp - Tm);
    s.gradh[a] = F2(0.5f) * (hp - hm);
    s.dLam[a] = upwind(s.u[a], lc - lm, lp - lc);
  }
  if constexpr (HD == kHandState) {
    s.P = w2(WP::P, o);
    s.cs2 = w2(WP::CS2, o);
    s.e = handed_energy(h, s.P, s.rho);
  } else {
    s.P = vdw_pressure(m, s.rho, s.T);
    s.cs2 = vdw_cs2(m, s.rho, s.T);
    s.e = EN ? e0 : vdw_energy(m, s.rho, s.T);
  }
  if (ODD && !two) {                                         // a lone last node: both halves are this node
    s.rho.y = s.rho.x;
    s.T.y = s.T.x;
    s.P.y = s.P.x;
  }
#pragma unroll
  for (int i = 0; i < L::Q; ++i) v[L::Q + i] = pulled(i, L::Q + i);
  Attractors<D, F2> at;
  at.setup(m, s);
  if (at.flags) atomicOr(err, at.flags);
  auto put = [&](const int i, const F2 val) {
    ST* Bi = at_bytes(B + (long long)i * p.plane, bo);
    if (!pop_ok(p, Bi, 0, 2)) return;
    if (two) Store<S>::st2_stream(Bi, val, p.ref[i]);
    else Store<S>::template st_stream<float>(Bi, 0, val.x, p.ref[i]);
  };
  FactoredRelax<D, F2>::f_pass(at, [&](int i) { return Store<S>::value(v[i], p.ref[i]); }, put);
  FactoredRelax<D, F2>::g_pass(at, [&](int i) { return Store<S>::value(v[L::Q + i], p.ref[L::Q + i]); },
                               [&](int i, F2 x) { put(L::Q + i, x); });
}
template <int D, typename S, Handed HD, bool ODD, int NTB, int MINB>
__global__ void __launch_bounds__(NTB, MINB)
k_collide2(const __grid_constant__ Params p, const NodeRange range, const typename Store<S>::T* __restrict__ A,
           typename Store<S>::T* __restrict__ B, const float* __restrict__ M, const float* __restrict__ W,
           unsigned* err) {
  wait_previous_launch();
  collide_pairs<D, S, HD, ODD, NTB, MINB>(p, range, A, B, M, W, err, blockIdx.x);
}

// ---------------------------------------------------------------------------
// ghost fill of the post-collision buffer (non-periodic x only): inflow faces
// get the stored equilibria of their state, outflow faces copy the nearest
// interior node, wall faces re-emit the mass that the nearest interior node
// sends into the wall with the equilibrium of the wall (diffuse reflection):
// s f^eq, s g^eq at (rho_e, u_wall, T_wall), rho_e that node's density, s =
// (its f with c_x towards the wall) / (the f^eq with c_x away from it).  Reads
// only the interior nodes next to the faces, so the rows may be filled in any
// order.
//
// The G ghost values of a row and direction are equal, so the work item is
// (face, direction, row): one load and one G-wide store, every item touching
// sectors of its own (no coalescing is possible: rows are a pitch apart).  A
// wall face takes (face, row) items instead, one equilibrium for the G layers
// of all directions.  Bound: one 32-byte sector read and one written per item;
// with an item per (layer, row) and a loop over the 2Q directions the fill of
// a 384x128x128 FP32 box was a chain of 54 dependent load-store pairs, 155 us
// against 73 us now; a 4096x2048 FP32 plane 13.4 against 5.1 us; the walls of a
// 100x24x20 FP64 channel 33 us (one FP64 equilibrium per layer) against 19 us.
// ---------------------------------------------------------------------------
template <int D, typename S>
__device__ __forceinline__ void ghost_store(const Params& p, typename Store<S>::T* B, long long o,
                                            typename Store<S>::T v) {
  using ST = typename Store<S>::T;
  static_assert(kGhost == 4, "four ghost layers");
  if (!pop_ok(p, B, o, kGhost)) return;
  constexpr int kVec = 16 / int(sizeof(ST)) < kGhost ? 16 / int(sizeof(ST)) : kGhost;   // values per store
  struct alignas(kVec * sizeof(ST)) Vec { ST v[kVec]; };
  if ((o & (kVec - 1)) == 0) {
    Vec w;
#pragma unroll
    for (int k = 0; k < kVec; ++k) w.v[k] = v;
#pragma unroll
    for (int k = 0; k < kGhost; k += kVec) *reinterpret_cast<Vec*>(B + o + k) = w;
  } else {
#pragma unroll
    for (int k = 0; k < kGhost; ++k) B[o + k] = v;
  }
}

// (One copy of the code for every kernel that fills walls: inlined, the compiler's choice
// of multiply-adds in the FP64 equilibrium differed, and a batch's walls with it.)
template <int D, typename S>
__device__ __noinline__ void ghost_wall_row(const Params& p, typename Store<S>::T* B, bool low, long long row) {
  using L = Lattice<D>;
  using ST = typename Store<S>::T;
  const long long o = row * p.pitch + (low ? 0 : p.Nx + p.G), os = row * p.pitch + (low ? p.G : p.G + p.Nx - 1);
  const int towards = low ? -1 : 1;
  double rho_e = 0.0, into = 0.0;
#pragma unroll
  for (int i = 0; i < L::Q; ++i) {
    const double v = pop_ok(p, B, i * p.plane + os) ? Store<S>::template ld<double>(B, i * p.plane + os, p.ref[i]) : 0.0;
    rho_e += v;
    if (L::c(i, 0) == towards) into += v;
  }
  const double* st = low ? p.st_lo : p.st_hi;
  double uw[D], feq[L::Q], geq[L::Q];
#pragma unroll
  for (int a = 0; a < D; ++a) uw[a] = st[1 + a];
  equilibria<D>(model_of<double>(p), rho_e, uw, st[4], feq, geq);
  double out = 0.0;
#pragma unroll
  for (int i = 0; i < L::Q; ++i)
    if (L::c(i, 0) == -towards) out += feq[i];
  const double s = into / out;
#pragma unroll
  for (int i = 0; i < L::Q; ++i) {
    ST f, g;
    Store<S>::template st<double>(&f, 0, s * feq[i], p.ref[i]);
    Store<S>::template st<double>(&g, 0, s * geq[i], p.ref[L::Q + i]);
    ghost_store<D, S>(p, B, i * p.plane + o, f);
    ghost_store<D, S>(p, B, (L::Q + i) * p.plane + o, g);
  }
}

// The ghost layers of row Br of population i of a bounded box from the row's own
// first / last node (outflow) or the face's equilibrium (inflow); `first`,
// `last`: the ends to fill.  The nodes may have been written by this block
// before a barrier, so they are read past L1.
template <int D, typename S>
__device__ __forceinline__ void ghost_row(const Params& p, typename Store<S>::T* Br, int i, bool first, bool last) {
  typename Store<S>::T v;
  if (first && pop_ok(p, Br, p.G)) {
    if (p.bc_lo == LBM_BC_INFLOW) Store<S>::template st<double>(&v, 0, p.eq_lo[i], p.ref[i]);
    else v = __ldcg(Br + p.G);
    ghost_store<D, S>(p, Br, 0, v);
  }
  if (last && pop_ok(p, Br, p.G + p.Nx - 1)) {
    if (p.bc_hi == LBM_BC_INFLOW) Store<S>::template st<double>(&v, 0, p.eq_hi[i], p.ref[i]);
    else v = __ldcg(Br + p.G + p.Nx - 1);
    ghost_store<D, S>(p, Br, p.G + p.Nx, v);
  }
}

// work items of the two faces: rows of a wall face, (direction, row) pairs of another
template <int D> __host__ __device__ inline long long ghost_items(const Params& p, bool low) {
  const long long rows = (long long)p.Ny * p.Nz;
  return (low ? p.bc_lo : p.bc_hi) == LBM_BC_WALL ? rows : rows * 2 * Lattice<D>::Q;
}

// items first, first + stride, ... of a handle whose x faces are not periodic
template <int D, typename S>
__device__ __forceinline__ void ghost_fill(const Params& p, typename Store<S>::T* B, long long first,
                                           long long stride) {
  using ST = typename Store<S>::T;
  const long long rows = (long long)p.Ny * p.Nz, nlo = ghost_items<D>(p, true), n = nlo + ghost_items<D>(p, false);
  for (long long it = first; it < n; it += stride) {
    const bool low = it < nlo;
    const long long k = low ? it : it - nlo;
    const int bc = low ? p.bc_lo : p.bc_hi;
    if (bc == LBM_BC_WALL) {
      ghost_wall_row<D, S>(p, B, low, k);
      continue;
    }
    const int i = int(k / rows);
    const long long b = i * p.plane + (k - i * rows) * p.pitch;
    ST v;
    if (bc == LBM_BC_INFLOW) {
      Store<S>::template st<double>(&v, 0, (low ? p.eq_lo : p.eq_hi)[i], p.ref[i]);
    } else {
      const long long os = b + (low ? p.G : p.G + p.Nx - 1);
      if (!pop_ok(p, B, os)) continue;
      v = B[os];
    }
    ghost_store<D, S>(p, B, b + (low ? 0 : p.Nx + p.G), v);
  }
}

// one item per thread; small blocks, so that the rows of a wall (an FP64
// equilibrium each) spread over the multiprocessors
constexpr int kGhostBlock = 64;
template <int D, typename S>
__global__ void __launch_bounds__(kGhostBlock) k_ghosts(const __grid_constant__ Params p, typename Store<S>::T* B) {
  wait_previous_launch();
  ghost_fill<D, S>(p, B, blockIdx.x * (long long)kGhostBlock + threadIdx.x, (long long)gridDim.x * kGhostBlock);
}

// ---------------------------------------------------------------------------
// split step, pass 3 in FP32 arithmetic with the rows staged in shared memory:
// a block owns W consecutive x of one row (y, z).  Its warps request every row
// segment the block reads (the 2Q pulled populations and the primitive fields of
// the row and of its neighbours along y and z) by bulk asynchronous copies, one
// per segment, completing on one mbarrier; each thread then collides two nodes
// from shared memory.  The loads hold no registers and no threads while they
// are in flight, and an operand address is a base plus a compile-time offset:
// with loads to registers a third of the instructions were 64-bit address
// arithmetic and 8 warps per multiprocessor waited on them.  256^3: 1437 us with
// loads to registers, 1619 us with copies issued lane by lane, 1158 us in this form
// and 1102 us (7.0 TB/s, the copy rate) since it reads fewer fields; FP16 deviations
// 873 and 790 us, bound by the issue of the conversions.
//
// Segments start at multiples of W elements of the padded row; in FP32 storage of a
// bounded row from its first node on (the G elements before it are a 16-byte unit),
// which saves rows of a multiple of W a segment of G nodes (256x128x96 with the
// learned closure: 784 -> 778 us per step).  A population
// with c_x = +1 needs the element left of the segment, one with c_x = -1 the
// element right of it: their segments are one 16-byte unit (kA elements) longer
// on that side.  On a periodic x the unit across the seam is a copy of its own,
// which needs Nx to be a multiple of the unit (collide_rows_ok).
// ---------------------------------------------------------------------------
constexpr unsigned kWaitLimit = 1u << 22;     // polls of a copy's completion before the step gives up

// Row segments of one block: element offsets in shared memory.
template <int D, typename S, Handed HD, int W> struct RowsLayout {
  using ST = typename Store<S>::T;
  static constexpr int Q = Lattice<D>::Q, T3 = Q / 3;            // directions per c_x
  static constexpr int kA = 16 / int(sizeof(ST)), kF = 4;        // elements per 16 bytes: populations, fields
  // populations of one kind: T3 rows of W + kA (c_x = -1), T3 of W, T3 of W + kA
  static constexpr int kSet = T3 * (3 * W + 2 * kA);
  __host__ __device__ static constexpr int row(int i) {
    return i < T3 ? i * (W + kA) : (i < 2 * T3 ? T3 * (W + kA) + (i - T3) * W : T3 * (2 * W + kA) + (i - 2 * T3) * (W + kA));
  }
  // index of the segment's first node in row i (the left unit of c_x = +1 rows)
  __host__ __device__ static constexpr int lead(int i) { return i < 2 * T3 ? 0 : kA; }
  // padded x of the first segment
  __host__ __device__ static constexpr int first(int G, bool bounded) { return bounded && G % kA == 0 ? G : 0; }
  static constexpr size_t kPopBytes = size_t(2 * kSet) * sizeof(ST);
  // field rows (planes of W): nWide of the row with a unit on both sides; then the
  // row's nOwn; then nSide of the two neighbours along each b > 0
  static constexpr bool DER = derives_fields<float, HD>();       // h, Lam_a from rho, u_a, T; else read
  static constexpr bool EN = HD == kHandEnergy;                  // e of every node read, for h
  static constexpr bool LAP = hands_laplacian<D, float>();       // F from the Laplacian; else read
  static constexpr int RHO = -1;                                 // the density, a plane of M
  static constexpr int nF = LAP ? 0 : D;
  static constexpr int nSide = (DER ? 3 : 4) + EN + LAP, nOwn = nF + D - 1 + (DER ? 0 : D);
  static constexpr int kWide = W + 2 * kF, nWide = nSide, nNb = 2 * nSide * (D - 1);
  // wide and side fields of axis a: u_a, T, then rho (and e), or h and Lam_a; the Laplacian
  static constexpr int kU = 0, kT = 1, kRho = 2, kEn = 3, kH = 2, kLam = 3, kLap = (DER ? 3 : 4) + EN;
  __host__ __device__ static constexpr int field(int a, int k) {
    using WP = WPlanes<D>;
    return k == kU ? WP::U + a : (k == kT ? WP::T : (k == kLap ? WP::F : (DER ? (k == kRho ? RHO : WP::E) : (k == kH ? WP::H : WP::LAM + a))));
  }
  // own rows: F_a, u_b (b > 0), then, if read, Lam_b (b > 0) and rho
  static constexpr int ownRho = nF + 2 * (D - 1);
  __host__ __device__ static constexpr int ownU(int b) { return nF + b - 1; }
  __host__ __device__ static constexpr int ownLam(int b) { return nF + D - 1 + b - 1; }
  __host__ __device__ static constexpr int own_field(int k) {
    using WP = WPlanes<D>;
    return k < nF ? WP::F + k : (k < ownLam(1) ? WP::U + 1 + k - nF : (k < ownRho ? WP::LAM + 1 + k - ownLam(1) : RHO));
  }
  __host__ __device__ static constexpr int wide(int k) { return k * kWide + kF; }
  __host__ __device__ static constexpr int own(int k) { return nWide * kWide + k * W; }
  __host__ __device__ static constexpr int nb(int b, int side, int k) {   // b in 1 .. D - 1, side 0 (minus) or 1 (plus)
    return nWide * kWide + (nOwn + ((b - 1) * 2 + side) * nSide + k) * W;
  }
  static constexpr int nRows = 2 * Q + nWide + nOwn + nNb;
  static constexpr size_t kBytes = kPopBytes + sizeof(float) * size_t(nWide * kWide + (nOwn + nNb) * W) + 16;
};

constexpr int kRowW = 128;                    // nodes of a block's segment

// segments of a row
template <typename S> inline int collide_segments(const Params& p) {
  constexpr int kA = 16 / int(sizeof(typename Store<S>::T));
  const int first = !p.periodic_x && p.G % kA == 0 ? p.G : 0;              // RowsLayout::first
  return (p.G + p.Nx - first + kRowW - 1) / kRowW;
}

// The row form applies when every seam unit is a whole 16-byte unit (4 FP32, 8
// FP16-deviation values), and is taken when the segments are full enough: its cost is
// per segment, k_collide2's per node.  Periodic rows cross at 9/16 (2 million nodes, us
// per step, rows and pairs: Nx 64 292 and 283, 72 317 and 338, 128 234 and 287, 136 301
// and 316; a box of 4 x 224 x 224: 375 and 170), in both storage types.  Bounded rows,
// whose ghosts the row form fills and whose pairs straddle 16-byte units, at 3/16 in FP32
// (Nx 16 964 and 929, 24 639 and 658, 128 307 and 422) and 1/4 with FP16 deviations (24
// 883 and 433, 32 513 and 546, 128 323 and 348); and whatever the fill while the segments
// are one round of blocks, for the launch that the ghosts take otherwise (17 x 16 x 16
// FP32: 16.6 and 19.0; 1225 segments of 16 nodes 18 and 17).
template <typename S> inline bool collide_rows_ok(const Params& p) {
  constexpr int kA = 16 / int(sizeof(typename Store<S>::T));
  if (p.periodic_x && p.Nx % kA) return false;
  if (!p.periodic_x && (long long)collide_segments<S>(p) * p.Ny * p.Nz <= 512) return true;
  const int sixteenths = p.periodic_x ? 9 : (kA == 4 ? 3 : 4);
  return 16 * p.Nx >= sixteenths * kRowW * collide_segments<S>(p);
}

__device__ __forceinline__ void bulk_copy(unsigned dst, const void* src, unsigned bytes, unsigned bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst),
               "l"(src), "r"(bytes), "r"(bar)
               : "memory");
}

// one thread of the (converged) warp
__device__ __forceinline__ bool elect_one() {
  unsigned e;
  asm volatile("{\n .reg .pred p;\n elect.sync _|p, 0xffffffff;\n selp.u32 %0, 1, 0, p;\n}\n" : "=r"(e));
  return e != 0;
}

template <int D, typename S, Handed HD, bool BOUNDED, int W, int MINB>
__device__ __forceinline__ void collide_rows(const Params& p, int nseg, FastDiv dseg, FastDiv dny, const typename Store<S>::T* __restrict__ A,
                                             typename Store<S>::T* __restrict__ B, const float* __restrict__ M,
                                             const float* __restrict__ Wf, unsigned* err, const unsigned block) {
  using L = Lattice<D>;
  using ST = typename Store<S>::T;
  using WP = WPlanes<D>;
  using R = RowsLayout<D, S, HD, W>;
  constexpr int Q = L::Q;
  extern __shared__ __align__(128) unsigned char smem_raw[];
  ST* sp = reinterpret_cast<ST*>(smem_raw);
  float* sf = reinterpret_cast<float*>(smem_raw + R::kPopBytes);
  uint64_t* bar = reinterpret_cast<uint64_t*>(smem_raw + R::kBytes - 16);
  const unsigned row = dseg.div(block), seg = block - row * unsigned(nseg);
  const int z = D == 3 ? int(dny.div(row)) : 0, y = int(row) - z * p.Ny;
  const int x0 = R::first(p.G, BOUNDED) + int(seg) * W, xend = BOUNDED ? p.pitch : p.Nx;        // padded x; end of the row's copied part
  const unsigned pitch = unsigned(p.pitch), r0 = row * pitch;
  // bytes of every segment with its side units (16 bytes each; absent at the
  // ends of a bounded row)
  const int n = min(W, xend - x0);                                     // elements of the segment itself
  const bool lseam = !BOUNDED && x0 == 0, rseam = !BOUNDED && x0 + W >= p.Nx;
  const bool lside = x0 > 0, rside = x0 + n < xend;                    // side units contiguous with the segment
  if (threadIdx.x == 0) {
    tc::mbar_init(bar, 1);
    const unsigned nl = BOUNDED ? unsigned(lside) : 1u, nr = BOUNDED ? unsigned(rside) : 1u;
    const unsigned bytes = unsigned(n) * (2u * Q * sizeof(ST) + 4u * (R::nWide + R::nOwn + R::nNb)) +
                           16u * (nl + nr) * (2u * R::T3 + R::nWide);
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(tc::smem_addr(bar)), "r"(bytes) : "memory");
  }
  __syncthreads();
  {
    // the warps take the segments in turn, one elected thread each: the
    // addresses are uniform, so a request costs a few instructions
    const unsigned s0 = tc::smem_addr(smem_raw), b0 = tc::smem_addr(bar);
    const int warp = __shfl_sync(0xffffffffu, int(threadIdx.x >> 5), 0);
    // (pop: a row of populations, checked)
    auto copy = [&](const bool pop, const unsigned d, const char* src, const unsigned bytes) {
#ifdef LBM_BOUNDS_CHECK
      const ST* e = reinterpret_cast<const ST*>(src);
      const int ne = int(bytes / sizeof(ST));
      if (pop && !pop_inside(p, e, 0, ne)) {
        ST* to = reinterpret_cast<ST*>(smem_raw + (d - s0));
        for (int k = 0; k < ne; ++k) to[k] = pop_value(p, e + k);
        asm volatile("mbarrier.complete_tx.relaxed.cta.shared::cta.b64 [%0], %1;" ::"r"(b0), "r"(bytes) : "memory");
        return;
      }
#endif
      bulk_copy(d, src, bytes, b0);
    };
    auto segment = [&](const bool pop, const void* rowp, const unsigned es, const unsigned dst, const bool left, const bool right) {
      const char* src = static_cast<const char*>(rowp) + (long long)x0 * es;
      const unsigned d = s0 + dst, nb = unsigned(n) * es;
      const unsigned l = left && lside ? 16u : 0u, r = right && rside ? 16u : 0u;
      copy(pop, d - l, src - l, nb + l + r);
      if (left && lseam) copy(pop, d - 16, static_cast<const char*>(rowp) + (long long)p.Nx * es - 16, 16);
      if (right && rseam) copy(pop, d + nb, static_cast<const char*>(rowp), 16);
    };
    if (elect_one()) {
      constexpr int NW = W / 64;
      const int ym = wrap(y - 1, p.Ny), yp = wrap(y + 1, p.Ny), zm = D == 3 ? wrap(z - 1, p.Nz) : 0, zp = D == 3 ? wrap(z + 1, p.Nz) : 0;
      auto rowof = [&](const int cy, const int cz) {                   // element offset of row (y + cy, z + cz)
        const int yy = cy < 0 ? ym : (cy > 0 ? yp : y), zz = D == 3 ? (cz < 0 ? zm : (cz > 0 ? zp : z)) : 0;
        return (long long)(zz * p.Ny + yy) * p.pitch;
      };
#pragma unroll
      for (int w = 0; w < NW; ++w) {
        if (warp != w) continue;
#pragma unroll
        for (int k = w; k < R::nRows; k += NW) {
          if (k < 2 * Q) {
            const int i = k < Q ? k : k - Q, cx = L::c(i, 0);
            const ST* rowp = A + (long long)k * p.plane + rowof(-L::c(i, 1), D == 3 ? -L::c(i, D - 1) : 0);
            segment(true, rowp, sizeof(ST), unsigned((k < Q ? 0 : R::kSet) + R::row(i) + R::lead(i)) * unsigned(sizeof(ST)), cx > 0, cx < 0);
          } else {
            int c = k - 2 * Q, f = 0, dst = 0, dy = 0, dz = 0;
            const bool wide = c < R::nWide;
            if (wide) {
              f = R::field(0, c);
              dst = R::wide(c);
            } else if (c < R::nWide + R::nOwn) {
              f = R::own_field(c - R::nWide);
              dst = R::own(c - R::nWide);
            } else {
              c -= R::nWide + R::nOwn;
              const int bb = 1 + c / (2 * R::nSide), side = (c / R::nSide) & 1, q = c % R::nSide;
              dst = R::nb(bb, side, q);
              f = R::field(bb, q);
              (bb == 1 ? dy : dz) = side ? 1 : -1;
            }
            segment(false, (f < 0 ? M : Wf + (long long)f * p.plane) + rowof(dy, dz), sizeof(float), unsigned(R::kPopBytes) + unsigned(dst) * 4u, wide, wide);
          }
        }
      }
    }
    __syncwarp();
  }
#ifdef LBM_BOUNDS_CHECK
  __syncthreads();                                                     // the elements copied by plain stores
#endif
  const int t = threadIdx.x, xp = x0 + 2 * t, xhi = p.G + p.Nx;
  const bool act = xp >= p.G && xp < xhi, two = xp + 1 < xhi;
  const unsigned o = r0 + unsigned(xp);
  const Model<float> m = model_of<float>(p);
  NodeState<D, F2> s;
  s.sc = p.sc_on != 0;
  s.mu_num = s.eta_num = s.k_num = F2(0.f);
  auto g2 = [&](const float* base, long long k) { return f2_of(__ldg(reinterpret_cast<const float2*>(base + k * p.plane + o))); };
  if (act) {
    if (s.sc) {
      const float* V = static_cast<const float*>(p.sc_visc);
      s.mu_num = g2(V, 0);
      s.eta_num = g2(V, 1);
      s.k_num = g2(V, 2);
    }
    if constexpr (HD == kHandState) {
      s.P = g2(Wf, WP::P);
      s.cs2 = g2(Wf, WP::CS2);
    }
  }
  const bool ok = tc::mbar_wait(bar, 0, kWaitLimit);
  if (!ok) {
    atomicOr(err, kFlagWait);
    tc::mbar_wait(bar, 0, kWaitLimit);                                 // the copies still in flight
  }
  if (ok && act) {
  auto f2at = [&](int off) { return f2_of(*reinterpret_cast<const float2*>(sf + off + 2 * t)); };
  auto f1at = [&](int off) { return sf[off + 2 * t]; };
  s.rho = f2at(R::DER ? R::wide(R::kRho) : R::own(R::ownRho));
  s.T = f2at(R::wide(R::kT));
  // h and theta = P / rho of a node pair from rho and T, and e where it is handed on
  auto enthalpy = [&](const F2 rho, const F2 T, const F2 e, F2& th) {
    const F2 hd = vdw_enthalpy(m, rho, T, th);
    return R::EN ? e + th : hd;
  };
  F2 h, theta, e0(0.f), e1(0.f);
  if constexpr (R::EN) e0 = f2at(R::wide(R::kEn));
  if constexpr (R::DER) h = enthalpy(s.rho, s.T, e0, theta);
  else h = f2at(R::wide(R::kH));
  const F2 kr = F2(m.kappa) * s.rho * F2(0.5f);
  s.div_u = F2(0.f);
#pragma unroll
  for (int a = 0; a < D; ++a) {
    s.u[a] = f2at(a == 0 ? R::wide(R::kU) : R::own(R::ownU(a)));
    if constexpr (!R::LAP) s.F[a] = f2at(R::own(a));
    F2 lc, up, um, Tp, Tm, hp, hm, lp, lm;
    if constexpr (R::DER) lc = lambda_of(s.rho, s.u[a], theta);
    else lc = f2at(a == 0 ? R::wide(R::kLam) : R::own(R::ownLam(a)));
    if (a == 0) {
      // outer neighbours of the pair: x - 1 and x + 2
      auto outer = [&](const int k) { return F2(f1at(R::wide(k) - 1), f1at(R::wide(k) + 2)); };
      const F2 uo = outer(R::kU), To = outer(R::kT);
      F2 ho, lo;
      if constexpr (R::DER) {
        const F2 ro = outer(R::kRho);
        F2 tho;
        if constexpr (R::EN) e1 = outer(R::kEn);
        ho = enthalpy(ro, To, e1, tho);
        lo = lambda_of(ro, uo, tho);
      } else {
        ho = outer(R::kH);
        lo = outer(R::kLam);
      }
      if constexpr (R::LAP) {
        const F2 c = f2at(R::wide(R::kLap)), n2 = outer(R::kLap);
        s.F[0] = kr * (F2(c.y, n2.y) - F2(n2.x, c.x));                                     // Eq. FK
      }
      up = F2(s.u[0].y, uo.y);
      um = F2(uo.x, s.u[0].x);
      Tp = F2(s.T.y, To.y);
      Tm = F2(To.x, s.T.x);
      hp = F2(h.y, ho.y);
      hm = F2(ho.x, h.x);
      lp = F2(lc.y, lo.y);
      lm = F2(lo.x, lc.x);
    } else {
      auto side = [&](const int d, const int k) { return f2at(R::nb(a, d, k)); };
      um = side(0, R::kU);
      up = side(1, R::kU);
      Tm = side(0, R::kT);
      Tp = side(1, R::kT);
      if constexpr (R::DER) {
        const F2 rm = side(0, R::kRho), rp = side(1, R::kRho);
        F2 th;
        if constexpr (R::EN) e1 = side(0, R::kEn);
        hm = enthalpy(rm, Tm, e1, th);
        lm = lambda_of(rm, um, th);
        if constexpr (R::EN) e1 = side(1, R::kEn);
        hp = enthalpy(rp, Tp, e1, th);
        lp = lambda_of(rp, up, th);
      } else {
        hm = side(0, R::kH);
        hp = side(1, R::kH);
        lm = side(0, R::kLam);
        lp = side(1, R::kLam);
      }
      if constexpr (R::LAP) s.F[a] = kr * (side(1, R::kLap) - side(0, R::kLap));
    }
    s.div_u = mad(F2(0.5f), up - um, s.div_u);
    s.gradT[a] = F2(0.5f) * (Tp - Tm);
    s.gradh[a] = F2(0.5f) * (hp - hm);
    s.dLam[a] = upwind(s.u[a], lc - lm, lp - lc);
  }
  if constexpr (HD == kHandState) {
    s.e = handed_energy(h, s.P, s.rho);
  } else {
    s.P = vdw_pressure(m, s.rho, s.T);
    s.cs2 = vdw_cs2(m, s.rho, s.T);
    s.e = R::EN ? e0 : vdw_energy(m, s.rho, s.T);
  }
  if (!two) {                                                          // a lone last node: both halves are this node
    s.rho.y = s.rho.x;
    s.T.y = s.T.x;
    s.P.y = s.P.x;
  }
  Attractors<D, F2> at;
  at.setup(m, s);
  if (at.flags) atomicOr(err, at.flags);
  // a row's pull of direction i: elements x - c_x of the pair
  auto pulled = [&](const int i, const int set) {
    const ST* q = sp + set + R::row(i) + R::lead(i) + 2 * t;
    const int cx = L::c(i, 0);
    return Store<S>::value(cx == 0 ? Store<S>::raw2s(q) : Store<S>::raw11s(q - cx), p.ref[set ? Q + i : i]);
  };
  auto put = [&](const int i, const F2 val) {
    ST* Bi = B + (long long)i * p.plane + o;
    if (!pop_ok(p, Bi, 0, 2)) return;
    const typename Store<S>::Raw q = Store<S>::pack(val, p.ref[i]);
    if (!BOUNDED || two) Store<S>::st2_raw(Bi, q);
    else Bi[0] = Store<S>::half_of(q, 0);
  };
  FactoredRelax<D, F2>::f_pass(at, [&](int i) { return pulled(i, 0); }, put);
  FactoredRelax<D, F2>::g_pass(at, [&](int i) { return pulled(i, R::kSet); }, [&](int i, F2 x) { put(Q + i, x); });
  }
  // ghost layers of a bounded row, by the blocks of its first and last node
  // (their sectors have just been written; a wall's equilibrium is k_ghosts')
  if constexpr (BOUNDED) {
    const bool first = seg == 0 && p.bc_lo != LBM_BC_WALL, last = xhi - 1 >= x0 && xhi - 1 < x0 + W && p.bc_hi != LBM_BC_WALL;
    if (first || last) {
      __syncthreads();
      for (int i = t; i < 2 * Q; i += W / 2) ghost_row<D, S>(p, B + (long long)i * p.plane + r0, i, first, last);
    }
  }
}
template <int D, typename S, Handed HD, bool BOUNDED, int W, int MINB>
__global__ void __launch_bounds__(W / 2, MINB)
k_collide_rows(const __grid_constant__ Params p, int nseg, FastDiv dseg, FastDiv dny,
               const typename Store<S>::T* __restrict__ A, typename Store<S>::T* __restrict__ B,
               const float* __restrict__ M, const float* __restrict__ Wf, unsigned* err) {
  wait_previous_launch();
  collide_rows<D, S, HD, BOUNDED, W, MINB>(p, nseg, dseg, dny, A, B, M, Wf, err, blockIdx.x);
}

// ---------------------------------------------------------------------------
// outputs: interior rho, u, T as FP64 (interior layout) and FP64 totals
// ---------------------------------------------------------------------------
template <int D, typename real>
__global__ void k_pack(Params p, const real* M, const real* W, double* rho, double* u, double* T) {
  int xp, y, z;
  if (!decode(p, blockIdx.x * (long long)blockDim.x + threadIdx.x, p.G, p.G + p.Nx, xp, y, z)) return;
  const long long o = node_off(p, xp, y, z);
  const long long N = (long long)p.Nx * p.Ny * p.Nz;
  const long long n = (xp - p.G) + (long long)p.Nx * (y + (long long)p.Ny * z);
  if (rho) rho[n] = double(M[o]);
  if (u)
    for (int a = 0; a < D; ++a) u[a * N + n] = double(W[a * p.plane + o]);
  if (T) T[n] = double(W[D * p.plane + o]);
}

// block partials of K sums per thread: warp-shuffle reduction, then one value per
// warp through shared memory
template <int K> __device__ __forceinline__ void block_partials(const double (&acc)[K], double* partials) {
  __shared__ double sh[32][K];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  for (int k = 0; k < K; ++k) {
    double v = acc[k];
    for (int off = 16; off > 0; off >>= 1) v += __shfl_down_sync(0xffffffffu, v, off);
    if (lane == 0) sh[warp][k] = v;
  }
  __syncthreads();
  if (threadIdx.x < K) {
    double v = 0.0;
    for (int w = 0; w < int(blockDim.x >> 5); ++w) v += sh[w][threadIdx.x];
    partials[blockIdx.x * K + threadIdx.x] = v;
  }
}

// block partials of (sum rho, sum (j + F/2), sum (S + u.F/2)) in FP64
template <int D, typename real>
__global__ void k_totals(Params p, const real* M, const real* W, double* partials) {
  constexpr int K = D + 2;
  double acc[K];
  for (int k = 0; k < K; ++k) acc[k] = 0.0;
  const long long n = (long long)p.Nx * p.Ny * p.Nz;
  for (long long gid = blockIdx.x * (long long)blockDim.x + threadIdx.x; gid < n;
       gid += (long long)gridDim.x * blockDim.x) {
    int xp, y, z;
    decode(p, gid, p.G, p.G + p.Nx, xp, y, z);
    const long long o = node_off(p, xp, y, z);
    acc[0] += double(M[o]);
    double uF = 0.0;
    for (int a = 0; a < D; ++a) {
      const double F = double(W[(2 * D + 2 + a) * p.plane + o]);
      acc[1 + a] += double(M[(1 + a) * p.plane + o]) + 0.5 * F;
      uF += double(W[a * p.plane + o]) * F;
    }
    acc[1 + D] += double(M[(1 + D) * p.plane + o]) + 0.5 * uF;
  }
  block_partials<K>(acc, partials);
}

// The same of FP32 fields, bound by the FP64 units when every value is converted and
// added in FP64 (28 such instructions per node).  A thread takes four nodes of a row at a
// time and sums them in FP32 without loss: the sum's rounding errors (two-sums, Knuth, The
// Art of Computer Programming 2, 4.2.2; products leave a remainder) are summed next to it,
// and their rounding errors in turn (the second-order form of Klein, "A generalized
// Kahan-Babuska-Summation-Algorithm", 2006); what is dropped is 2^-72 of the sum.  FP64
// joins the three once per thread.  A thread that met an infinity, a NaN or FP32's range
// (its sums are then not finite) adds its nodes again in FP64.
// 384x128x128: 77 us, 800x800 18 us; all in FP64 296 and 35; with FP64 additions for each
// group of four and the errors in FP32 alone (2^-48) 58 and 16.
struct Sum3 {                                                    // two lanes
  F2 s = F2(0.f), e = F2(0.f), r = F2(0.f);
  __device__ __forceinline__ void error(F2 v) {
    F2 b;
    e = two_sum(e, v, b);
    r = r + b;
  }
  __device__ __forceinline__ void add(F2 v) {
    F2 a;
    s = two_sum(s, v, a);
    error(a);
  }
  __device__ __forceinline__ bool finite() const { return isfinite((s.x + s.y) + (e.x + e.y)); }
  __device__ __forceinline__ double value() const {
    float a, b, c;                                               // the lanes joined without loss first
    const float t = two_sum(s.x, s.y, a), u = two_sum(e.x, e.y, b), w = two_sum(u, a, c);
    return double(t) + (double(w) + double((r.x + r.y) + (b + c)));
  }
};
template <int D>
__global__ void __launch_bounds__(256) k_totals_row(const __grid_constant__ Params p, const NodeRange range,
                                                    const float* __restrict__ M, const float* __restrict__ W,
                                                    double* partials) {
  using WP = WPlanes<D>;
  constexpr int K = D + 2;
  Sum3 sum[K];
  for (unsigned gid = blockIdx.x * 256u + threadIdx.x; gid < range.n; gid += gridDim.x * 256u) {
    int xp, y, z;
    range.decode(gid, xp, y, z);
    const unsigned o = (unsigned(z) * unsigned(p.Ny) + unsigned(y)) * unsigned(p.pitch) + unsigned(xp);
    bool in[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) in[k] = xp + k >= p.G && xp + k < p.G + p.Nx;
    auto load = [&](const float* plane, F2 (&v)[2]) {            // nodes outside the box count as zeros
      const float4 q = __ldg(reinterpret_cast<const float4*>(plane + o));
      v[0] = F2(in[0] ? q.x : 0.f, in[1] ? q.y : 0.f);
      v[1] = F2(in[2] ? q.z : 0.f, in[3] ? q.w : 0.f);
    };
    F2 v[2], w[2], u[2], F[2];
    load(M, v);
    load(M + (1 + D) * p.plane, w);
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      sum[0].add(v[q]);
      sum[1 + D].add(w[q]);
    }
#pragma unroll
    for (int a = 0; a < D; ++a) {                                // j + F / 2; S + u . F / 2
      load(M + (1 + a) * p.plane, v);
      load(W + (WP::F + a) * p.plane, F);
      load(W + (WP::U + a) * p.plane, u);
#pragma unroll
      for (int q = 0; q < 2; ++q) {
        const F2 h = F2(0.5f) * F[q], m = u[q] * h;
        sum[1 + a].add(v[q]);
        sum[1 + a].add(h);
        sum[1 + D].add(m);
        sum[1 + D].error(mad(u[q], h, F2(-1.f) * m));
      }
    }
  }
  double acc[K];
  bool finite = true;
#pragma unroll
  for (int k = 0; k < K; ++k) {
    acc[k] = sum[k].value();
    finite = finite && sum[k].finite();
  }
  if (!finite) {
#pragma unroll
    for (int k = 0; k < K; ++k) acc[k] = 0.0;
    for (unsigned gid = blockIdx.x * 256u + threadIdx.x; gid < range.n; gid += gridDim.x * 256u) {
      int xp, y, z;
      range.decode(gid, xp, y, z);
      const unsigned o = (unsigned(z) * unsigned(p.Ny) + unsigned(y)) * unsigned(p.pitch);
      for (int x = max(xp, p.G); x < min(xp + 4, p.G + p.Nx); ++x) {
        double uF = 0.0;
        acc[0] += double(M[o + x]);
#pragma unroll
        for (int a = 0; a < D; ++a) {
          const double f = double(W[(WP::F + a) * p.plane + o + x]);
          acc[1 + a] += double(M[(1 + a) * p.plane + o + x]) + 0.5 * f;
          uF += double(W[(WP::U + a) * p.plane + o + x]) * f;
        }
        acc[1 + D] += double(M[(1 + D) * p.plane + o + x]) + 0.5 * uF;
      }
    }
  }
  block_partials<K>(acc, partials);
}

// sum of the block partials in a fixed order: one warp per component, 32 strided
// partial sums and a butterfly (one thread per component took 57 us for 1024
// blocks, a chain of dependent loads; 3 us now)
template <int D>
__global__ void __launch_bounds__(32 * (D + 2)) k_totals_final(const double* partials, int nblocks, double* totals) {
  constexpr int K = D + 2;
  const int k = threadIdx.x >> 5, lane = threadIdx.x & 31;
  double v = 0.0;
  for (int b = lane; b < nblocks; b += 32) v += partials[b * K + k];
#pragma unroll
  for (int d = 16; d > 0; d >>= 1) v += __shfl_xor_sync(0xffffffffu, v, d);
  if (lane == 0) totals[k] = v;
}

}  // namespace lbm
