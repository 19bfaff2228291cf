// lbm_tile2d.cuh - the 2-D step: one launch, one tile of the plane per block.
//
// A block of threads owns a tile of TX x TY nodes, one unit per thread (two
// neighbouring nodes in packed FP32 arithmetic, one node in FP64), and does
// everything of Sec. 3.2 between reading the post-collision populations of the
// last step and writing the new ones:
//   A. every thread pulls the 2Q populations of its unit and keeps them; the
//      units of the halo (radius 3 in the L1 norm) are shared out: f only (rho),
//      f and g on radius 1 (j, S)
//   B. Laplacian of rho on radius 2
//   C. Korteweg force and primitive fields on radius 1
//   D. derivatives and collision of the unit from the populations kept in A.
// A population of a tile node is read once, the new ones are written once; the
// halo costs 9 reads per unit of radius 3 and arithmetic, all of it next to the
// tile's own lines.  Marching rows through a ring (the form before) re-read every
// population for the collision and had three barriers for every row of 128
// nodes.  Ghost layers of bounded rows are filled by the blocks that own the
// first and the last node (wall faces by k_ghosts).  Per launch, that form and this:
// 4096x2048 FP32 531 and 343 us (FP32 latency at 16 warps per multiprocessor), 800x800
// 90 and 32 us, 1000x4 FP64 198 and 18.5 us.
#pragma once

#include "lbm_kernels.cuh"
#include "lbm_closure.cuh"

namespace lbm {

// S = |grad u + grad u^T| / 2 and |grad s| of shock capturing (lbm_n1.cuh) from
// the central differences g[a][b] = d_a u_b, d_a T, d_a rho and rho, T
template <int D, typename C, typename V>
__device__ __forceinline__ void n1_norms(const Model<C>& m, const V (&g)[D][D], const V (&gT)[D], const V (&gr)[D],
                                         V rho, V T, V& S, V& gs) {
  V acc = V(0);
#pragma unroll
  for (int a = 0; a < D; ++a)
#pragma unroll
    for (int b = 0; b < D; ++b) acc = mad(g[a][b] + g[b][a], g[a][b] + g[b][a], acc);
  S = V(C(0.5)) * root(acc);
  V cT, cR;
  entropy_coefs(m, rho, T, cT, cR);
  V s2 = V(0);
#pragma unroll
  for (int a = 0; a < D; ++a) {
    const V d = mad(cT, gT[a], V(-1) * (cR * gr[a]));
    s2 = mad(d, d, s2);
  }
  gs = root(s2);
}

// One unit of nodes along x and its arithmetic.
template <typename S, typename real> struct Unit;
template <typename S> struct Unit<S, float> {          // two nodes, packed
  static constexpr int N = 2;
  using ST = typename Store<S>::T;
  using V = F2;
  using Raw = typename Store<S>::Raw;
  // byte offsets of x - 1, x, x + 1, x + 2; vec: x even and x + 1 next to it
  struct X { unsigned m, c, p, q; bool vec; };
  template <class Map> __device__ static X offsets(const Map& map, int gx) {
    constexpr unsigned E = sizeof(ST);
    X x;
    x.m = map(gx - 1) * E;
    x.c = map(gx) * E;
    x.p = map(gx + 1) * E;
    x.q = map(gx + 2) * E;
    x.vec = (x.c & E) == 0 && x.p == x.c + E;
    return x;
  }
  __device__ static Raw pull(const ST* row, int cx, const X& x) {
    if (cx > 0) return Store<S>::raw11(at_bytes(row, x.m), at_bytes(row, x.c));
    if (cx < 0) return Store<S>::raw11(at_bytes(row, x.p), at_bytes(row, x.q));
    return x.vec ? Store<S>::raw2g(at_bytes(row, x.c)) : Store<S>::raw11(at_bytes(row, x.c), at_bytes(row, x.p));
  }
  // the same with every element checked
  __device__ static Raw pull_checked(const Params& p, const ST* row, int cx, const X& x) {
    const unsigned a = cx > 0 ? x.m : (cx < 0 ? x.p : x.c), b = cx > 0 ? x.c : (cx < 0 ? x.q : x.p);
    return Store<S>::raw_of(pop_value(p, at_bytes(row, a)), pop_value(p, at_bytes(row, b)));
  }
  __device__ static V value(Raw r, float ref) { return Store<S>::value(r, ref); }
  __device__ static V ld(const float* s) { return f2_of(*reinterpret_cast<const float2*>(s)); }
  __device__ static void st(float* s, V v) { *reinterpret_cast<float2*>(s) = f2_in(v); }
  __device__ static V left(const float* s, V c) { return F2(s[-1], c.x); }       // values at x - 1 of the nodes
  __device__ static V right(const float* s, V c) { return F2(c.y, s[2]); }
  __device__ static float get(V v, int k) { return k ? v.y : v.x; }
  __device__ static void set(V& v, int k, float a) { (k ? v.y : v.x) = a; }
  __device__ static void store(ST* p, V v, float ref, bool two) {
    const Raw q = Store<S>::pack(v, ref);
    if (two) Store<S>::st2_raw(p, q);
    else p[0] = Store<S>::half_of(q, 0);
  }
  // values at x - 2 .. x + 2 of the nodes of the unit at s
  __device__ static void five(const float* s, V (&w)[5]) {
    w[0] = ld(s - 2);
    w[2] = ld(s);
    w[4] = ld(s + 2);
    w[1] = F2(w[0].y, w[2].x);
    w[3] = F2(w[2].y, w[4].x);
  }
  __device__ static V ld_field(const float* p) { return f2_of(__ldg(reinterpret_cast<const float2*>(p))); }
  __device__ static void store_field(float* p, V v, bool two) {
    if (two) *reinterpret_cast<float2*>(p) = f2_in(v);
    else p[0] = v.x;
  }
};
template <typename S> struct Unit<S, double> {         // one node
  static constexpr int N = 1;
  using ST = typename Store<S>::T;
  using V = double;
  using Raw = double;
  struct X { unsigned m, c, p; };
  template <class Map> __device__ static X offsets(const Map& map, int gx) {
    constexpr unsigned E = sizeof(ST);
    return {map(gx - 1) * E, map(gx) * E, map(gx + 1) * E};
  }
  __device__ static Raw pull(const ST* row, int cx, const X& x) {
    return double(__ldg(at_bytes(row, cx > 0 ? x.m : (cx < 0 ? x.p : x.c))));
  }
  __device__ static Raw pull_checked(const Params& p, const ST* row, int cx, const X& x) {
    return double(pop_value(p, at_bytes(row, cx > 0 ? x.m : (cx < 0 ? x.p : x.c))));
  }
  __device__ static V value(Raw r, float) { return r; }
  __device__ static V ld(const double* s) { return *s; }
  __device__ static void st(double* s, V v) { *s = v; }
  __device__ static V left(const double* s, V) { return s[-1]; }
  __device__ static V right(const double* s, V) { return s[1]; }
  __device__ static double get(V v, int) { return v; }
  __device__ static void set(V& v, int, double a) { v = a; }
  __device__ static void store(ST* p, V v, float ref, bool) { Store<S>::template st_stream<double>(p, 0, v, ref); }
  __device__ static void five(const double* s, V (&w)[5]) {
#pragma unroll
    for (int k = 0; k < 5; ++k) w[k] = s[k - 2];
  }
  __device__ static V ld_field(const double* p) { return __ldg(p); }
  __device__ static void store_field(double* p, V v, bool) { *p = v; }
};

// Shared-memory boxes of a tile: density (radius 3), Laplacian (radius 2),
// primitive fields (radius 1: u, T, h, Lam; the halo's j and S stand in the
// places of u and T until stage C), own density of a wall's ghost columns.
template <typename real, int N, int TX, int TY> struct TileGeom {
  static constexpr int U3 = (3 + N - 1) / N, U2 = (2 + N - 1) / N, U1 = 1;     // halo units along x
  static constexpr int NT = TX / N * TY;
  static constexpr int P3 = TX + 2 * U3 * N, P2 = TX + 2 * U2 * N, P1 = TX + 2 * U1 * N;   // row lengths (nodes)
  static constexpr int H3 = TY + 6, H2 = TY + 4, H1 = TY + 2;
  static constexpr int PU = 0, PT = 2, PH = 3, PL = 4, NPRM = 6;
  static constexpr int oLap = P3 * H3, oPrm = oLap + P2 * H2, oOwn = oPrm + NPRM * P1 * H1, kElems = oOwn + 2 * H1;
  static constexpr size_t kBytes = (sizeof(real) * size_t(kElems) + 15) & ~size_t(15);
  static_assert(NT % 32 == 0, "whole warps");
};

// units of a box of `units` x `rows` outside the inner `iu` x `ir` box (`hu`
// units and `hr` rows of halo): unit k of the ring as (unit, row) of the box
struct Ring {
  int units, rows, hu, hr;
  __device__ __forceinline__ int count() const { return units * rows - (units - 2 * hu) * (rows - 2 * hr); }
  __device__ __forceinline__ void at(int k, int& u, int& r) const {
    const int band = units * hr;
    if (k < 2 * band) {                                 // rows below, rows above
      const int q = k / units;
      u = k - q * units;
      r = q < hr ? q : rows - 2 * hr + q;
      return;
    }
    k -= 2 * band;                                      // the sides of the inner rows
    const int q = k / (2 * hu), c = k - q * 2 * hu;
    u = c < hu ? c : units - 2 * hu + c;
    r = hr + q;
  }
};

// kNorms: with shock capturing on, leave S and |grad s| for k_n1_coef_2d
// HELP: threads of the block beyond the tile's units.  They take the halo first,
// next to the warps that own the units: where a small plane leaves a block a
// multiprocessor of its own, its time is the chain of loads and divisions of a
// unit, not their number (FP64 1000x4: 26 us with the owners doing the halo
// after their own units, 18.5 us now).
template <typename S, typename real, class CL, int TX, int TY, int HELP, bool kNorms>
__device__ __forceinline__ void tile2d(const Params& p, const typename Store<S>::T* __restrict__ A,
                                       typename Store<S>::T* __restrict__ B, const int x0, const int y0, real* sm,
                                       unsigned& flags, const CL& closure) {
  using L = Lattice<2>;
  using ST = typename Store<S>::T;
  using U = Unit<S, real>;
  using V = typename U::V;
  constexpr int N = U::N, Q = L::Q;
  using G = TileGeom<real, N, TX, TY>;
  real *s_rho = sm, *s_lap = sm + G::oLap, *s_prm = sm + G::oPrm, *s_own = sm + G::oOwn;
  constexpr int NTB = G::NT + HELP;
  const int tid = threadIdx.x, ux = tid % (TX / N), uy = tid / (TX / N);
  const bool own = HELP == 0 || tid < G::NT;
  const int rank = HELP == 0 ? tid : (own ? tid + HELP : tid - G::NT);       // order in which the halo is taken
  const Model<real> m = model_of<real>(p);
  const bool wtile = (p.bc_lo == LBM_BC_WALL && x0 < 4) || (p.bc_hi == LBM_BC_WALL && x0 + TX + 4 > p.Nx);
  // padded x of any box coordinate: wrapped (images past the seam are the nodes
  // themselves) or, on a bounded x, kept inside the row (values past the ghost
  // layers are not used)
  auto map = [&](int gx) -> unsigned {
    if (p.periodic_x) {
      gx += gx < 0 ? p.Nx : 0;
      gx -= gx >= p.Nx ? p.Nx : 0;
      if (unsigned(gx) >= unsigned(p.Nx)) {             // a box wider than the domain
        gx %= p.Nx;
        gx += gx < 0 ? p.Nx : 0;
      }
      return unsigned(gx);
    }
    return unsigned(min(max(gx + p.G, 0), p.pitch - 1));
  };
  auto row = [&](int gy) -> unsigned {
    gy += gy < 0 ? p.Ny : 0;
    gy -= gy >= p.Ny ? p.Ny : 0;
    if (unsigned(gy) >= unsigned(p.Ny)) {
      gy %= p.Ny;
      gy += gy < 0 ? p.Ny : 0;
    }
    return unsigned(gy) * unsigned(p.pitch) * unsigned(sizeof(ST));
  };
  // populations of direction set `set` (0: f, Q: g) of the unit at (gx, gy)
  auto pull_set = [&](const typename U::X& x, const unsigned (&r)[3], const int set, typename U::Raw* v) {
#pragma unroll
    for (int i = 0; i < Q; ++i) {
      const ST* Ai = A + (long long)(set + i) * p.plane;
      const ST* rp = at_bytes(Ai, r[L::c(i, 1) + 1]);
#ifdef LBM_BOUNDS_CHECK
      v[i] = U::pull_checked(p, rp, L::c(i, 0), x);
#else
      v[i] = U::pull(rp, L::c(i, 0), x);
#endif
    }
  };
  auto rows3 = [&](int gy, unsigned (&r)[3]) {
#pragma unroll
    for (int c = -1; c <= 1; ++c) r[c + 1] = row(gy - c);
  };
  // density and momentum sums (j exactly zero for mirror-symmetric populations)
  auto sums = [&](const typename U::Raw* v, V& rho, V* j) {
    V sp[2] = {V(0), V(0)}, sn[2] = {V(0), V(0)};
    rho = V(0);
#pragma unroll
    for (int i = 0; i < Q; ++i) {
      const V w = U::value(v[i], p.ref[i]);
      rho += w;
#pragma unroll
      for (int a = 0; a < 2; ++a) {
        if (L::c(i, a) == 1) sp[a] += w;
        if (L::c(i, a) == -1) sn[a] += w;
      }
    }
#pragma unroll
    for (int a = 0; a < 2; ++a) j[a] = sp[a] - sn[a];
  };
  auto energy = [&](const typename U::Raw* v) {
    V s = V(0);
#pragma unroll
    for (int i = 0; i < Q; ++i) s += U::value(v[i], p.ref[Q + i]);
    return s;
  };
  // density that the Laplacian reads at the unit: ghost columns of a wall face
  // hold their mirror image's, their own goes to s_own (columns -1 and Nx)
  auto capillary = [&](V rho, int gx, int gy, int r1) {
    if (wtile) {
#pragma unroll
      for (int k = 0; k < N; ++k) {
        const int x = gx + k, xw = wall_mirror(p, x);
        if (xw == x) continue;
        if ((x == -1 || x == p.Nx) && r1 >= 0 && r1 < G::H1) s_own[(x < 0 ? 0 : G::H1) + r1] = U::get(rho, k);
        real q = real(0);
        if (xw >= -3 && xw <= p.Nx + 2) {
#pragma unroll
          for (int i = 0; i < Q; ++i) {
            const ST* Ai = A + (long long)i * p.plane;
            const ST* v = at_bytes(Ai, row(gy - L::c(i, 1)) + map(xw - L::c(i, 0)) * unsigned(sizeof(ST)));
            q += pop_ok(p, v, 0) ? Store<S>::template ld<real>(v, 0, p.ref[i]) : real(0);
          }
        }
        U::set(rho, k, q);
      }
    }
    return rho;
  };

  // ---------------- A: the thread's own unit, then its share of the halo -------
  const int gx = x0 + N * ux, gy = y0 + uy;
  const typename U::X xo = U::offsets(map, gx);
  unsigned ro[3];
  rows3(gy, ro);
  typename U::Raw f[Q], g[Q];
  if (own) {
    pull_set(xo, ro, 0, f);
    pull_set(xo, ro, Q, g);
  }
  const Ring ring3{G::P3 / N, G::H3, G::U3, 3};
  for (int k = rank; k < ring3.count(); k += NTB) {
    int bu, br;
    ring3.at(k, bu, br);
    const int hx = x0 + N * (bu - G::U3), hy = y0 + br - 3;
    // distance of the unit's nearest node from the tile
    const int dx = hx < x0 ? x0 - hx - (N - 1) : (hx >= x0 + TX ? hx - (x0 + TX) + 1 : 0);
    const int dy = br < 3 ? 3 - br : (br >= TY + 3 ? br - TY - 2 : 0);
    if (dx + dy > 3) continue;
    const typename U::X hxo = U::offsets(map, hx);
    unsigned hr[3];
    rows3(hy, hr);
    typename U::Raw v[Q];
    pull_set(hxo, hr, 0, v);
    V rho, j[2];
    sums(v, rho, j);
    U::st(s_rho + br * G::P3 + N * bu, capillary(rho, hx, hy, br - 2));
    if (dx + dy <= 1) {
      pull_set(hxo, hr, Q, v);
      real* d = s_prm + (br - 2) * G::P1 + N * (bu - G::U3 + G::U1);
      U::st(d, j[0]);
      U::st(d + G::P1 * G::H1, j[1]);
      U::st(d + 2 * G::P1 * G::H1, energy(v));
    }
  }
  V rho, j[2], Se = V(0);
  if (own) {
    sums(f, rho, j);
    Se = energy(g);
    U::st(s_rho + (uy + 3) * G::P3 + N * (ux + G::U3), wtile ? capillary(rho, gx, gy, uy + 1) : rho);
  }
  __syncthreads();

  // ---------------- B: Laplacian of rho on radius 2 ----------------------------
  for (int k = tid; k < G::P2 / N * G::H2; k += NTB) {
    const int br = k / (G::P2 / N), bu = k - br * (G::P2 / N);
    const real* r = s_rho + (br + 1) * G::P3 + N * (bu + G::U3 - G::U2);
    const V c = U::ld(r), c2 = c + c;
    const V lap = ((U::right(r, c) + U::left(r, c)) - c2) + ((U::ld(r + G::P3) + U::ld(r - G::P3)) - c2);
    U::st(s_lap + br * G::P2 + N * bu, lap);
  }
  __syncthreads();

  // ---------------- C: force and primitive fields on radius 1 ------------------
  // unit (bu, br) of the radius-1 box with its moments; returns rho-independent
  // results through F, T (and P, c_s^2 of closures that hand them on)
  auto prims = [&](int bu, int br, V rho, const V* j, V Sg, bool act, V* F, V* u, V& T, V& P, V& cs2, V& e) {
    const real* l = s_lap + (br + 1) * G::P2 + N * (bu + G::U2 - G::U1);
    const V kr = V(m.kappa) * rho * V(real(0.5)), lc = U::ld(l);
    F[0] = kr * (U::right(l, lc) - U::left(l, lc));                                      // Eq. FK
    F[1] = kr * (U::ld(l + G::P2) - U::ld(l - G::P2));
    V uF = V(0), u2 = V(0);
    e = V(0);
    const Divider<V> over_rho(rho);
#pragma unroll
    for (int a = 0; a < 2; ++a) {
      u[a] = over_rho(mad(V(real(0.5)), F[a], j[a]));                                    // Eq. def_u
      uF = mad(u[a], F[a], uF);
      u2 = mad(u[a], u[a], u2);
    }
    const V E = over_rho(mad(V(real(0.5)), uF, Sg));                                     // Eq. def_E
#pragma unroll
    for (int k = 0; k < N; ++k) {
      real t = real(0), pp = real(1), c = real(0), ee = real(0);
      if (CL::kWarp || act) closure(m, U::get(rho, k), U::get(E, k), U::get(u2, k), act, t, pp, c, ee);
      U::set(T, k, t);
      U::set(P, k, pp);
      U::set(cs2, k, c);
      U::set(e, k, ee);
    }
    if (!act) return;
    const V theta = P / rho, w = V(real(3)) * (theta - V(real(1.0 / 3.0)));
    real* d = s_prm + br * G::P1 + N * bu;
    auto put = [&](int k, V v) { U::st(d + k * G::P1 * G::H1, v); };
#pragma unroll
    for (int a = 0; a < 2; ++a) {
      const V ru = rho * u[a];
      put(G::PU + a, u[a]);
      put(G::PL + a, mad(ru * u[a], u[a], w * ru));
    }
    put(G::PT, T);
    put(G::PH, e + theta);                                                               // Eq. enthalpy
  };
  const Ring ring1{G::P1 / N, G::H1, G::U1, 1};
  for (int k = rank; CL::kWarp ? k - (tid & 31) < ring1.count() : k < ring1.count(); k += NTB) {
    int bu = 0, br = 0;
    if (k < ring1.count()) ring1.at(k, bu, br);
    const bool corner = (br == 0 || br == G::H1 - 1) && (bu == 0 || bu == G::P1 / N - 1);
    const bool act = k < ring1.count() && !corner;
    if (!CL::kWarp && !act) continue;
    V hr = V(1), hj[2] = {V(0), V(0)}, hS = V(0), F[2], u[2], T, P, cs2, e;
    if (act) {
      hr = U::ld(s_rho + (br + 2) * G::P3 + N * (bu + G::U3 - G::U1));
      if (wtile) {
#pragma unroll
        for (int q = 0; q < N; ++q) {
          const int x = x0 + N * (bu - G::U1) + q;
          if (wall_mirror(p, x) != x && (x == -1 || x == p.Nx)) U::set(hr, q, s_own[(x < 0 ? 0 : G::H1) + br]);
        }
      }
      const real* d = s_prm + br * G::P1 + N * bu;
      hj[0] = U::ld(d);
      hj[1] = U::ld(d + G::P1 * G::H1);
      hS = U::ld(d + 2 * G::P1 * G::H1);
    }
    prims(bu, br, hr, hj, hS, act, F, u, T, P, cs2, e);
  }
  NodeState<2, V> s;
  s.rho = rho;
  V e0 = V(0);
  if (own) prims(ux + G::U1, uy + 1, rho, j, Se, true, s.F, s.u, s.T, s.P, s.cs2, e0);
  __syncthreads();

  // ---------------- D: derivatives and collision -------------------------------
  const bool act = own && gx < p.Nx && gy < p.Ny, two = gx + N - 1 < p.Nx;
  if (act) {
    const unsigned o = unsigned(gy) * unsigned(p.pitch) + unsigned(gx + p.G);
    s.sc = p.sc_on != 0;
    s.mu_num = s.eta_num = s.k_num = V(0);
    if (s.sc) {
      const real* Vc = static_cast<const real*>(p.sc_visc) + o;
      s.mu_num = U::ld(Vc);
      s.eta_num = U::ld(Vc + p.plane);
      s.k_num = U::ld(Vc + 2 * p.plane);
    }
    const real* d = s_prm + (uy + 1) * G::P1 + N * (ux + G::U1);
    auto fld = [&](int k) { return d + k * G::P1 * G::H1; };
    if (s.sc) {
      // this step's fields for the shock-capturing coefficients of the next step:
      // rho and T with S and |grad s| (kNorms), or with u for the batched stencils
      const V half = V(real(0.5));
      real* W = static_cast<real*>(p.sc_prims) + o;
      U::store_field(W, s.rho, two);
      U::store_field(W + 3 * p.plane, s.T, two);
      if constexpr (kNorms) {
        // differences at the box ends are one-sided sums over the clamped node
        const bool lo = !p.periodic_x && gx == 0;
        auto diff = [&](const real* c, V v, int pitch, V gu[2]) {
          V r = U::right(c, v), l = U::left(c, v);
          if (lo) U::set(l, 0, U::get(v, 0));
#pragma unroll
          for (int q = 0; q < N; ++q)
            if (!p.periodic_x && gx + q == p.Nx - 1) U::set(r, q, U::get(v, q));
          gu[0] = half * (r - l);
          gu[1] = half * (U::ld(c + pitch) - U::ld(c - pitch));
        };
        V gu[2][2], gT[2], gr[2], t[2], Sn, gn;
#pragma unroll
        for (int b = 0; b < 2; ++b) {
          diff(fld(G::PU + b), s.u[b], G::P1, t);
          gu[0][b] = t[0];
          gu[1][b] = t[1];
        }
        diff(fld(G::PT), s.T, G::P1, gT);
        diff(s_rho + (uy + 3) * G::P3 + N * (ux + G::U3), s.rho, G::P3, gr);
        n1_norms<2>(m, gu, gT, gr, s.rho, s.T, Sn, gn);
        real* w0 = static_cast<real*>(const_cast<void*>(p.sc_visc)) + 3 * p.plane + o;
        U::store_field(w0, Sn, two);
        U::store_field(w0 + p.plane, gn, two);
      } else {
#pragma unroll
        for (int a = 0; a < 2; ++a) U::store_field(W + (1 + a) * p.plane, s.u[a], two);
      }
    }
    const V h = U::ld(fld(G::PH));
    if constexpr (CL::kExtra > 0) s.e = h - s.P / s.rho;
    else s.e = CL::kEnergy ? e0 : vdw_energy(m, s.rho, s.T);
    s.div_u = V(0);
    const V half = V(real(0.5));
#pragma unroll
    for (int a = 0; a < 2; ++a) {
      auto plus = [&](int k, V c) { return a == 0 ? U::right(fld(k), c) : U::ld(fld(k) + G::P1); };
      auto minus = [&](int k, V c) { return a == 0 ? U::left(fld(k), c) : U::ld(fld(k) - G::P1); };
      const V lc = U::ld(fld(G::PL + a));
      s.div_u = mad(half, plus(G::PU + a, s.u[a]) - minus(G::PU + a, s.u[a]), s.div_u);
      s.gradT[a] = half * (plus(G::PT, s.T) - minus(G::PT, s.T));
      s.gradh[a] = half * (plus(G::PH, h) - minus(G::PH, h));
      s.dLam[a] = upwind(s.u[a], lc - minus(G::PL + a, lc), plus(G::PL + a, lc) - lc);
    }
    if constexpr (N == 2) {
      if (!two) {                                       // a lone last node: both halves are this node
        U::set(s.rho, 1, U::get(s.rho, 0));
        U::set(s.T, 1, U::get(s.T, 0));
        U::set(s.P, 1, U::get(s.P, 0));
      }
    }
    Attractors<2, V> at;
    at.setup(m, s);
    flags |= at.flags;
    auto put = [&](const int i, const V v) {
      ST* Bi = B + (long long)i * p.plane + o;
      if (pop_ok(p, Bi, 0, N)) U::store(Bi, v, p.ref[i], two);
    };
    FactoredRelax<2, V>::f_pass(at, [&](int i) { return U::value(f[i], p.ref[i]); }, put);
    FactoredRelax<2, V>::g_pass(at, [&](int i) { return U::value(g[i], p.ref[Q + i]); },
                                [&](int i, V v) { put(Q + i, v); });
  }
  if (!p.periodic_x) {
    const bool first = x0 == 0 && p.bc_lo != LBM_BC_WALL, last = x0 <= p.Nx - 1 && p.Nx - 1 < x0 + TX && p.bc_hi != LBM_BC_WALL;
    if (first || last) {
      __syncthreads();                                  // the tile's new populations are written
      for (int k = tid; k < 2 * Q * TY; k += NTB) {
        const int i = k / TY, y = y0 + k - i * TY;
        if (y < p.Ny) ghost_row<2, S>(p, B + (long long)i * p.plane + (long long)y * p.pitch, i, first, last);
      }
    }
  }
}

template <typename S, typename real, class CL, int TX, int TY, int HELP, int MINB>
__global__ void __launch_bounds__(TX / Unit<S, real>::N * TY + HELP, MINB)
k_step2d(const __grid_constant__ Params p, const typename Store<S>::T* __restrict__ A,
         typename Store<S>::T* __restrict__ B, unsigned* err, int ntx) {
  wait_previous_launch();
  extern __shared__ __align__(128) unsigned char smem_raw[];
  using G = TileGeom<real, Unit<S, real>::N, TX, TY>;
  CL closure;
  closure.load(p, smem_raw + G::kBytes);                // (stage A's barrier covers it)
  unsigned flags = 0;
  tile2d<S, real, CL, TX, TY, HELP, true>(p, A, B, int(blockIdx.x % unsigned(ntx)) * TX, int(blockIdx.x / unsigned(ntx)) * TY,
                              reinterpret_cast<real*>(smem_raw), flags, closure);
  if (flags) atomicOr(err, flags);
}

// One instance of a batch: its parameters and its two population buffers.
struct BatchInstance {
  Params p;
  void* pop[2];
};

// One work item of a 2-D batch step: an instance's tile.
struct BatchItem {
  int inst, x0, y0;
};

// Batched step: the blocks are the tiles of every instance, largest instances
// first; `parity` selects which buffer of each instance is the source.
template <typename S, typename real, int TX, int TY, int MINB>
__global__ void __launch_bounds__(TX / Unit<S, real>::N * TY, MINB)
k_step2d_batch(const BatchInstance* __restrict__ insts, const BatchItem* __restrict__ items, int parity,
               unsigned* errs) {
  wait_previous_launch();
  extern __shared__ __align__(128) unsigned char smem_raw[];
  using ST = typename Store<S>::T;
  const BatchItem it = items[blockIdx.x];
  const BatchInstance& bi = insts[it.inst];
  unsigned flags = 0;
  tile2d<S, real, ExactClosure<real>, TX, TY, 0, false>(bi.p, reinterpret_cast<const ST*>(bi.pop[parity]),
                                              reinterpret_cast<ST*>(bi.pop[parity ^ 1]), it.x0, it.y0,
                                              reinterpret_cast<real*>(smem_raw), flags, ExactClosure<real>{});
  if (flags) atomicOr(errs + it.inst, flags);
}

// Batched fill of wall ghosts: the blocks of grid row k refill the wall faces of
// instance k, as k_ghosts does for one handle (other faces: the step itself).
template <int D, typename S>
__global__ void k_ghosts_batch(const BatchInstance* __restrict__ insts, int parity) {
  wait_previous_launch();
  using ST = typename Store<S>::T;
  const BatchInstance& bi = insts[blockIdx.y];
  const Params& p = bi.p;
  if (p.periodic_x || (p.bc_lo != LBM_BC_WALL && p.bc_hi != LBM_BC_WALL)) return;   // (an instance with launches of its own fills its walls after this)
  ghost_fill<D, S>(p, reinterpret_cast<ST*>(bi.pop[parity ^ 1]), blockIdx.x * (long long)blockDim.x + threadIdx.x,
                   (long long)gridDim.x * blockDim.x);
}

}  // namespace lbm
