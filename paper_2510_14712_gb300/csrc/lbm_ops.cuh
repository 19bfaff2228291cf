// lbm_ops.cuh - launch wrappers of one (D, storage, arithmetic) kernel set.
// Each k_*.cu translation unit instantiates one of them.
#pragma once

#include <type_traits>

#include <algorithm>
#include <vector>

#include "lbm_batch3d.cuh"

namespace lbm {

constexpr int kBlock = 256;

inline unsigned grid_for(long long n) { return unsigned((n + kBlock - 1) / kBlock); }

template <int D, typename S, typename real> struct OpsImpl {
  using ST = typename Store<S>::T;

  static real* M(Handle& h) { return reinterpret_cast<real*>(h.scratch); }
  static real* W(Handle& h) { return reinterpret_cast<real*>(h.scratch) + (D + 2) * h.p.plane; }

  static void init(Handle& h, const double* rho, const double* u, const double* T) {
    const Params& p = h.p;
    ST* A = reinterpret_cast<ST*>(h.pop[h.cur]);
    if constexpr (sizeof(real) == 4) {
      const NodeRange r = p.periodic_x ? NodeRange(p, 0, p.Nx) : NodeRange(p, -p.G - 1, p.Nx + p.G + 1);
      k_init_df<D, S><<<unsigned((r.n + 255u) / 256u), 128, 0, h.stream>>>(p, InitConsts(p), r, A, rho, u, T);
    } else {
      const long long n = (long long)(p.periodic_x ? p.Nx : p.Nx + 2 * p.G + 2) * p.Ny * p.Nz;
      k_init<D, S><<<unsigned((n + 127) / 128), 128, 0, h.stream>>>(p, A, rho, u, T);
    }
    h.launches += 1;
  }

  // moments of `src` into scratch
  static void moments(Handle& h, const void* src) {
    const Params& p = h.p;
    int lo, hi;
    moment_range(p, 3, lo, hi);
    const ST* A = reinterpret_cast<const ST*>(src);
    if constexpr (sizeof(real) == 4) {
      // groups start at multiples of 16 bytes of the padded row
      constexpr int N = Store<S>::kGroup;
      const NodeRange r(p, 0, p.Nx + 2 * p.G, N);
      auto kern = p.Nx % N ? k_moments_row<D, S, true> : k_moments_row<D, S, false>;
      launch_overlapped(kern, dim3(unsigned((r.n + 127u) / 128u)), 128, 0, h.stream, p, r, A, M(h));
    } else {
      const NodeRange r(p, lo, hi);
      launch_overlapped(k_moments<D>, dim3(grid_for(r.n)), kBlock, 0, h.stream, p, r, A, M(h));
    }
    h.launches += 1;
  }

  // blocks of k_prims3 per multiprocessor: 40 registers without a network
  template <class CL> static constexpr int kPrimsMinB = CL::kWarp ? 2 : (sizeof(real) == 8 ? 3 : 6);

  // z-segments of the columns of k_prims3: about one round of resident blocks over all
  // columns of the launch (a segment repeats four planes of density and two of
  // Laplacian), at least two planes each
  static int prim_segments(const Params& p, int slots, long long columns) {
    return int(std::max(1LL, std::min((long long)(p.Nz / 2), (slots + columns - 1) / columns)));
  }

  // primitive fields from the moments in scratch (3-D: MINB blocks per
  // multiprocessor for the register budget)
  template <class CL, int MINB = kPrimsMinB<CL>> static void prims(Handle& h) {
    const Params& p = h.p;
    int lo, hi;
    moment_range(p, 1, lo, hi);
    if constexpr (D == 3) {
      auto kern = k_prims3<real, CL, MINB>;
      const int slots = prepared_blocks<k_prims3<real, CL, MINB>>(kPrimX * kPrimY, CL::kSmem);
      const int ncolx = (hi - lo + kPrimX - 1) / kPrimX, ncoly = (p.Ny + kPrimY - 1) / kPrimY;
      const int nseg = prim_segments(p, slots, (long long)ncolx * ncoly);
      launch_overlapped(kern, dim3(unsigned(ncolx * ncoly * nseg)), kPrimX * kPrimY, CL::kSmem, h.stream, p, lo, hi, ncolx, ncoly, nseg,
                                                                                      M(h), W(h));
    } else {
      const NodeRange r(p, lo, hi);
      launch_overlapped(k_prims<D, real, CL>, dim3(grid_for(r.n)), kBlock, CL::kSmem, h.stream, p, r, M(h), W(h));
    }
    h.launches += 1;
  }

  // moments + primitive fields of `src` into scratch
  static void fields(Handle& h, const void* src) {
    moments(h, src);
    prims<AnyClosure<real>>(h);
  }

  // registers of the collision by rows: blocks per multiprocessor that the shared memory
  // admits (FP32: five of 40 KB, 1013 -> 990 us at 384x128x128 against the bound of 128
  // registers, which spilled; FP16 deviations: eight of 25 KB, 1234 us at 256^3, with
  // seven 1247); threads and blocks of the other forms
  static constexpr int kRowsMinB = sizeof(ST) == 4 ? 5 : 8, kColThreads = 128, kColMinB = 2;

  // collision of every interior node; whether it filled the ghost layers too
  template <Handed HD> static bool collide(Handle& h, const void* src, void* dst) {
    const Params& p = h.p;
    const ST* A = reinterpret_cast<const ST*>(src);
    ST* B = reinterpret_cast<ST*>(dst);
    h.launches += 1;
    if constexpr (sizeof(real) == 4) {
      if (collide_rows_ok<S>(p)) {
        constexpr int W128 = kRowW;
        using R = RowsLayout<D, S, HD, W128>;
        auto kern = p.periodic_x ? k_collide_rows<D, S, HD, false, W128, kRowsMinB> : k_collide_rows<D, S, HD, true, W128, kRowsMinB>;
        if (p.periodic_x) prepared_blocks<k_collide_rows<D, S, HD, false, W128, kRowsMinB>>(W128 / 2, R::kBytes);
        else prepared_blocks<k_collide_rows<D, S, HD, true, W128, kRowsMinB>>(W128 / 2, R::kBytes);
        const int nseg = collide_segments<S>(p);
        launch_overlapped(kern, dim3(unsigned(nseg) * unsigned(p.Ny) * unsigned(p.Nz)), W128 / 2, R::kBytes, h.stream,
            p, nseg, FastDiv(unsigned(nseg)), FastDiv(unsigned(p.Ny)), A, B, M(h), W(h), h.err_dev);
        return p.bc_lo != LBM_BC_WALL && p.bc_hi != LBM_BC_WALL;
      }
      constexpr int NTB = kColThreads, MINB = kColMinB;
      const NodeRange r(p, p.G, p.G + p.Nx, 2);
      auto kern = p.Nx % 2 ? k_collide2<D, S, HD, true, NTB, MINB> : k_collide2<D, S, HD, false, NTB, MINB>;
      launch_overlapped(kern, dim3(unsigned((r.n + NTB - 1) / NTB)), NTB, 0, h.stream, p, r, A, B, M(h), W(h), h.err_dev);
    } else {
      constexpr int NTB = kColThreads, MINB = kColMinB;
      const NodeRange r(p, p.G, p.G + p.Nx);
      launch_overlapped(k_collide<D, S, real, HD, NTB, MINB>, dim3(unsigned((r.n + NTB - 1) / NTB)), NTB, 0, h.stream, p, r, A, B, M(h),
                                                                                                W(h), h.err_dev);
    }
    return false;
  }

  // One step in three passes over the box: moments, primitive fields, collision.
  template <class CL, int MINB = kPrimsMinB<CL>> static void split(Handle& h, const void* src, void* dst) {
    moments(h, src);
    prims<CL, MINB>(h);
    if (!collide<handed<CL>()>(h, src, dst)) ghosts(h, dst);
  }

  static int multiprocessors() {
    static const int sms = [] {
      int n = 1, dev = 0;
      cudaGetDevice(&dev);
      cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev);
      return n;
    }();
    return sms;
  }

  // wall ghosts after a step whose kernel filled the other faces' layers
  static void wall_ghosts(Handle& h, void* dst) {
    if (h.p.bc_lo == LBM_BC_WALL || h.p.bc_hi == LBM_BC_WALL) ghosts(h, dst);
  }

  // One tile shape of the 2-D step (TX x TY nodes per block, MINB blocks per
  // multiprocessor for the register budget, HELP threads beyond the tile's units)
  // with thermodynamic closure CL.
  template <int TX, int TY, int MINB, class CL, int HELP = 0> struct Tile {
    using G = TileGeom<real, Unit<S, real>::N, TX, TY>;
    static constexpr size_t kSmem = G::kBytes + CL::kSmem;
    static long long tiles(const Params& p) {
      return (long long)((p.Nx + TX - 1) / TX) * ((p.Ny + TY - 1) / TY);
    }
    // work of a block in units of one population sum: density of the radius-3
    // box, primitive fields of the radius-1 box, collision of the tile
    static double work() { return G::P3 * G::H3 * 1.0 + G::P1 * G::H1 * 6.0 + TX * TY * 20.0; }
    static void launch(Handle& h, const void* src, void* dst) {
      const Params& p = h.p;
      auto kern = k_step2d<S, real, CL, TX, TY, HELP, MINB>;
      prepared_blocks<k_step2d<S, real, CL, TX, TY, HELP, MINB>>(G::NT + HELP, kSmem);
      launch_overlapped(kern, dim3(unsigned(tiles(p))), G::NT + HELP, kSmem, h.stream, p, reinterpret_cast<const ST*>(src), reinterpret_cast<ST*>(dst),
                                                          h.err_dev, (p.Nx + TX - 1) / TX);
      h.launches += 1;
      wall_ghosts(h, dst);
    }
  };

  // Candidate forms of the step, first = default.
  //
  // 3-D boxes take the split step: a kernel that marched columns with everything in
  // one pass evaluated the moments on 2.1 times the nodes (radius 3 around a 32x8
  // tile) and held 16 warps per multiprocessor behind three barriers a plane.  Per
  // step, that form and now: 256^3 FP32 2587 and 1808 us, FP16 deviations 2072 and
  // 1235 us, 91x75x53 FP32 129 and 67 us, Peng-Robinson 128^3 449 and 275 us, FP64
  // channel 100x24x20 1061 and 128 us, 256x128x96 with a network 1441 and 778 us.
  //
  // 2-D planes take one tile per block, the default picks the shape; FP64 planes of
  // 2^20 nodes and more the split step: a tile evaluates the density on twice its nodes,
  // which the FP64 units, not the memory, pay for (tiles and split step, us per step:
  // 256x256 85 and 68, 512x512 256 and 227, 1024x1024 988 and 865, 2048x2048 3921 and
  // 3423, where the row-marching form before took 3551).  Smaller planes, faster than
  // that form either way, keep the one launch that their batches share; a batch takes
  // planes that split in launches of their own, for the bits of a handle.
  static bool plane_splits(const Params& p) {
    return D == 2 && sizeof(real) == 8 && (long long)p.Nx * p.Ny >= (1 << 20);
  }
  using LaunchFn = void (*)(Handle&, const void*, void*);
  template <class CL> static int candidates(const LaunchFn** fns) {
    if constexpr (D == 3 && CL::kWarp) {
      // the network's registers: 128 and two blocks per multiprocessor, or one block
      // without spills (256x128x96: 778 and 785 us per step)
      static const LaunchFn c[] = {&split<CL, 2>, &split<CL, 1>};
      *fns = c;
      return 2;
    } else if constexpr (D == 3) {
      static const LaunchFn c[] = {&split<CL>};
      *fns = c;
      return 1;
    } else {
      return Tiles<CL>::list(fns);
    }
  }

  // The shapes of the 2-D step and the rule among them: blocks run in rounds of
  // one per multiprocessor, so the shape with the smallest rounds x work per
  // block is taken; large tiles (least halo) where there are many, small ones
  // where large ones would leave multiprocessors without a tile.
  template <class CL, class... T> struct TileSet {
    static constexpr int n = int(sizeof...(T));
    static void rule(Handle& h, const void* src, void* dst) {
      if constexpr (sizeof(real) == 8) {
        if (plane_splits(h.p)) return split<CL>(h, src, dst);
      }
      static const LaunchFn fn[] = {&T::launch...};
      const double work[] = {T::work()...};
      const long long tiles[] = {T::tiles(h.p)...};
      int best = 0;
      double bt = 1e300;
      for (int k = 0; k < n; ++k) {
        const double t = double((tiles[k] + multiprocessors() - 1) / multiprocessors()) * work[k];
        if (t < bt) {
          bt = t;
          best = k;
        }
      }
      fn[best](h, src, dst);
    }
    static int list(const LaunchFn** fns) {
      static const LaunchFn c[] = {&rule, &T::launch...};
      *fns = c;
      return n + 1;
    }
  };
  template <class CL, bool F64 = sizeof(real) == 8> struct Tiles
      : TileSet<CL, Tile<64, 8, CL::kWarp ? 1 : 2, CL>, Tile<64, 4, 4, CL>, Tile<32, 8, 4, CL>,
                Tile<16, 8, 8, CL>> {};
  template <class CL> struct Tiles<CL, true>
      : TileSet<CL, Tile<32, 8, 1, CL>, Tile<32, 4, 2, CL>, Tile<16, 4, 2, CL, 64>, Tile<16, 2, 2, CL, 96>,
                Tile<8, 4, 2, CL, 96>> {};

  static void ghosts(Handle& h, void* dst) {
    const Params& p = h.p;
    if (!p.periodic_x) {
      const long long n = ghost_items<D>(p, true) + ghost_items<D>(p, false);
      launch_overlapped(k_ghosts<D, S>, dim3(unsigned((n + kGhostBlock - 1) / kGhostBlock)), kGhostBlock, 0, h.stream,
          p, reinterpret_cast<ST*>(dst));
      h.launches += 1;
    }
  }

  // shock capturing: numerical mu, eta, k for the next step from this step's
  // rho, u (D planes), T (null: the 2-D step left S and |grad s|)
  static void shock_capturing(Handle& h, const real* rho, const real* u, const real* T) {
    h.launches += n1_update<D, S, real>(h.p, h.stream, rho, u, T);
  }

  // Indices of lbm_set_tile: the forms, repeated up to the number of shapes that the
  // lattice, precision and closure ever had, so that an index that was valid stays valid.
  template <class CL> static int indices(int n) {
    constexpr int had = CL::kPr ? 1 : (D == 3 ? (sizeof(real) == 8 ? 1 : (CL::kWarp ? 4 : 5)) : (sizeof(real) == 4 && !CL::kWarp ? 9 : 5));
    return std::max(n, had);
  }

  template <class CL> static void step_cl(Handle& h, const void* src, void* dst) {
    const LaunchFn* fns;
    const int n = candidates<CL>(&fns);
    const int cfg = h.tile_cfg < indices<CL>(n) ? h.tile_cfg % n : 0;
    fns[cfg](h, src, dst);
    if (h.p.sc_on && (D == 3 || (cfg == 0 && plane_splits(h.p)))) {
      shock_capturing(h, M(h), W(h), W(h) + D * h.p.plane);
    } else if (h.p.sc_on) {
      shock_capturing(h, nullptr, nullptr, nullptr);
    }
  }
  static void step(Handle& h, const void* src, void* dst) { step_cl<ExactClosure<real>>(h, src, dst); }

  // Time every candidate shape for `reps` steps from the current state into
  // the spare buffer (the state is not advanced) and keep the fastest.
  template <class CL> static int autotune_cl(Handle& h, int reps, float* best_ms) {
    const LaunchFn* fns;
    const int n = candidates<CL>(&fns);
    cudaEvent_t e0, e1;
    cudaEventCreate(&e0);
    cudaEventCreate(&e1);
    int best = 0;
    float bt = 1e30f;
    const void* src = h.pop[h.cur];
    void* dst = h.pop[h.cur ^ 1];
    for (int c = 0; c < n; ++c) {
      fns[c](h, src, dst);                                   // warm-up / occupancy query
      cudaEventRecord(e0, h.stream);
      for (int r = 0; r < reps; ++r) fns[c](h, src, dst);
      cudaEventRecord(e1, h.stream);
      cudaEventSynchronize(e1);
      float ms = 0.f;
      cudaEventElapsedTime(&ms, e0, e1);
      if (c < kMaxTiles) h.tune_ms[c] = ms / (reps > 0 ? reps : 1);
      if (ms < bt) {
        bt = ms;
        best = c;
      }
    }
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    h.tile_cfg = best;
    h.tune_n = std::min(indices<CL>(n), kMaxTiles);
    for (int c = n; c < h.tune_n; ++c) h.tune_ms[c] = h.tune_ms[c % n];
    if (best_ms) *best_ms = bt / (reps > 0 ? reps : 1);
    return best;
  }
  static int autotune(Handle& h, int reps, float* best_ms) { return autotune_cl<ExactClosure<real>>(h, reps, best_ms); }
  template <class CL> static int ntiles_cl() {
    const LaunchFn* fns;
    return indices<CL>(candidates<CL>(&fns));
  }
  static int ntiles() { return ntiles_cl<ExactClosure<real>>(); }

  static void step_multipass(Handle& h, const void* src, void* dst) {
    const Params& p = h.p;
    if (p.eos_kind == LBM_EOS_PR) {
      if constexpr (std::is_same<S, Fp16Dev>::value) return;   // refused at create
      else if (sizeof(real) == 4 && p.t64) split<PrClosure<real, true>>(h, src, dst);
      else split<PrClosure<real>>(h, src, dst);
    } else if (sizeof(real) == 4 && p.t64) {
      split<ExactClosure<real, true>>(h, src, dst);
    } else {
      split<ExactClosure<real>>(h, src, dst);
    }
    if (p.sc_on) shock_capturing(h, M(h), W(h), W(h) + D * p.plane);
  }

  static void macro(Handle& h, const void* src, double* rho, double* u, double* T, double* totals) {
    const Params& p = h.p;
    fields(h, src);
    const long long n = (long long)p.Nx * p.Ny * p.Nz;
    if (rho || u || T) {
      k_pack<D, real><<<grid_for(n), kBlock, 0, h.stream>>>(p, M(h), W(h), rho, u, T);
      h.launches += 1;
    }
    if (totals) {
      int nb;
      if constexpr (sizeof(real) == 4) {
        const NodeRange r(p, 0, p.Nx + 2 * p.G, 4);
        nb = std::min(int((r.n + kBlock - 1) / kBlock), kMaxPartials);
        k_totals_row<D><<<nb, kBlock, 0, h.stream>>>(p, r, M(h), W(h), h.partials);
      } else {
        nb = int(std::min((n + kBlock - 1) / kBlock, (long long)kMaxPartials));
        k_totals<D, real><<<nb, kBlock, 0, h.stream>>>(p, M(h), W(h), h.partials);
      }
      k_totals_final<D><<<1, 32 * (D + 2), 0, h.stream>>>(h.partials, nb, totals);
      h.launches += 2;
    }
  }

  // moments (D + 2 planes), primitive fields (3 D + 2, and P, c_s^2 for the
  // closures that hand them on: Peng-Robinson, or a network attached to FP32)
  static size_t scratch_bytes(const Params& p) {
    const int extra = p.eos_kind == LBM_EOS_PR || std::is_same<S, float>::value ? 2 : 0;
    return size_t(4 * D + 4 + extra) * size_t(p.plane) * sizeof(real);
  }

  // ---- batches -------------------------------------------------------------
  // instances that step with launches of their own: planes that a single handle splits
  // (a batch gives a handle's bits), and a 3-D batch of one
  static bool own_launches(const Batch& b, const Params& p) { return D == 2 ? plane_splits(p) : b.n == 1; }
  static void enqueue_own(Batch& b, int parity) {
    for (int k = 0; k < b.n; ++k) {
      Handle& h = *b.inst[k];
      if (!own_launches(b, h.p)) continue;
      const Handle saved = h;
      h.stream = b.stream;
      h.err_dev = b.d_errs + k;
      split<ExactClosure<real>>(h, h.pop[parity], h.pop[parity ^ 1]);
      if (h.p.sc_on && !b.tuning) shock_capturing(h, M(h), W(h), W(h) + D * h.p.plane);
      b.launches += h.launches - saved.launches;
      h = saved;
    }
  }

  // 2-D: one launch over the tiles of every instance
  template <int TX, int TY, int MINB> struct BatchTiles {
    using G = TileGeom<real, Unit<S, real>::N, TX, TY>;
    static int prepare(Batch& b) {
      std::vector<BatchInstance> ti(b.n);
      std::vector<BatchItem> items;
      std::vector<int> order(b.n), rowstart(b.n + 1, 0);      // rows of the batched shock-capturing kernels
      for (int k = 0; k < b.n; ++k) {
        const Handle& h = *b.inst[k];
        ti[k].p = h.p;
        ti[k].pop[0] = h.pop[0];
        ti[k].pop[1] = h.pop[1];
        order[k] = k;
        rowstart[k + 1] = rowstart[k] + (h.p.sc_on && !own_launches(b, h.p) ? h.p.Ny * h.p.Nz : 0);
      }
      std::stable_sort(order.begin(), order.end(), [&](int a, int c) {
        return (long long)ti[a].p.Nx * ti[a].p.Ny > (long long)ti[c].p.Nx * ti[c].p.Ny;
      });
      for (int k : order) {
        if (own_launches(b, ti[k].p)) continue;
        for (int y = 0; y < ti[k].p.Ny; y += TY)
          for (int x = 0; x < ti[k].p.Nx; x += TX) items.push_back({k, x, y});
      }
      if (b.d_insts) cudaFree(b.d_insts);
      if (b.d_items) cudaFree(b.d_items);
      if (b.d_n1rows) cudaFree(b.d_n1rows);
      b.d_insts = b.d_items = nullptr;
      b.d_n1rows = nullptr;
      if (dev_malloc(&b.d_insts, sizeof(BatchInstance) * b.n) != cudaSuccess) return LBM_ENOMEM;
      if (dev_malloc(&b.d_items, sizeof(BatchItem) * std::max<size_t>(items.size(), 1)) != cudaSuccess) return LBM_ENOMEM;
      if (dev_malloc(&b.d_n1rows, sizeof(int) * (b.n + 1)) != cudaSuccess) return LBM_ENOMEM;
      cudaMemcpy(b.d_insts, ti.data(), sizeof(BatchInstance) * b.n, cudaMemcpyHostToDevice);
      cudaMemcpy(b.d_items, items.data(), sizeof(BatchItem) * items.size(), cudaMemcpyHostToDevice);
      cudaMemcpy(b.d_n1rows, rowstart.data(), sizeof(int) * (b.n + 1), cudaMemcpyHostToDevice);
      b.n1rows = rowstart[b.n];
      b.nitems = int(items.size());
      // blocks per instance of the wall fill: one item per thread of the instance with the most
      long long ng = 0;
      for (int k = 0; k < b.n; ++k)
        if (!own_launches(b, ti[k].p) && (ti[k].p.bc_lo == LBM_BC_WALL || ti[k].p.bc_hi == LBM_BC_WALL))
          ng = std::max(ng, ghost_items<D>(ti[k].p, true) + ghost_items<D>(ti[k].p, false));
      b.ghost_blocks = unsigned(std::max(1LL, std::min((ng + 255) / 256, 4096LL)));
      cudaFuncSetAttribute(k_step2d_batch<S, real, TX, TY, MINB>, cudaFuncAttributeMaxDynamicSharedMemorySize, int(G::kBytes));
      return cudaGetLastError() == cudaSuccess ? LBM_OK : LBM_ECUDA;
    }
    static void enqueue(Batch& b, int parity) {
      const BatchInstance* insts = reinterpret_cast<const BatchInstance*>(b.d_insts);
      if (b.nitems > 0) {
        launch_overlapped(k_step2d_batch<S, real, TX, TY, MINB>, dim3(unsigned(b.nitems)), G::NT, G::kBytes, b.stream,
            insts, reinterpret_cast<const BatchItem*>(b.d_items), parity, b.d_errs);
        b.launches += 1;
        for (int k0 = 0; k0 < b.n; k0 += 65535) {
          launch_overlapped(k_ghosts_batch<D, S>, dim3(b.ghost_blocks, unsigned(b.n - k0 < 65535 ? b.n - k0 : 65535)), 256, 0, b.stream,
              insts + k0, parity);
          b.launches += 1;
        }
      }
      if (b.n1rows > 0 && !b.tuning) b.launches += n1_update_batch<real>(insts, b.d_n1rows, b.n, b.n1rows, b.stream);
      enqueue_own(b, parity);
    }
  };

  // 3-D: the passes of the split step, each one launch over the blocks of every instance
  // (one launch for each kind of instance that a pass distinguishes)
  struct BatchSplit {
    using Inst = SplitInstance<real>;
    using CL = ExactClosure<real>;
    static constexpr int kMinB = kPrimsMinB<CL>;
    // groups of work items
    enum { kMoments, kMomentsRagged, kPrims, kRows, kRowsBounded, kNodes, kNodesOdd, kStrain, kCoef };
    static_assert(kCoef + 2 == sizeof(Batch::group) / sizeof(int), "first items of the groups and their end");

    static int prepare(Batch& b) {
      std::vector<Inst> ti(b.n);
      std::vector<int> order;
      long long columns = 0, n1columns = 0, ng = 0;
      using N1 = N1Column<S, real>;
      for (int k = 0; k < b.n; ++k) {
        Handle& h = *b.inst[k];
        const Params& p = h.p;
        Inst& t = ti[k];
        t.ghosts = 0;
        if (own_launches(b, p)) continue;
        order.push_back(k);
        t.p = p;
        t.pop[0] = h.pop[0];
        t.pop[1] = h.pop[1];
        t.M = M(h);
        t.W = W(h);
        int lo, hi;
        moment_range(p, 3, lo, hi);
        if constexpr (sizeof(real) == 4) {
          t.moments = NodeRange(p, 0, p.Nx + 2 * p.G, Store<S>::kGroup);
          t.nodes = NodeRange(p, p.G, p.G + p.Nx, 2);
          t.rowseg = collide_rows_ok<S>(p) ? collide_segments<S>(p) : 0;
        } else {
          t.moments = NodeRange(p, lo, hi);
          t.nodes = NodeRange(p, p.G, p.G + p.Nx);
          t.rowseg = 0;
        }
        t.drowseg = FastDiv(unsigned(std::max(1, t.rowseg)));
        t.dny = FastDiv(unsigned(p.Ny));
        const bool wall = p.bc_lo == LBM_BC_WALL || p.bc_hi == LBM_BC_WALL;
        t.ghosts = !p.periodic_x && (wall || t.rowseg == 0);
        if (t.ghosts) ng = std::max(ng, ghost_items<D>(p, true) + ghost_items<D>(p, false));
        moment_range(p, 1, t.lo, t.hi);
        t.ncolx = (t.hi - t.lo + kPrimX - 1) / kPrimX;
        t.ncoly = (p.Ny + kPrimY - 1) / kPrimY;
        columns += (long long)t.ncolx * t.ncoly;
        const unsigned nx = unsigned((p.Nx + N1::N - 1) / N1::N);
        t.units = p.sc_on ? nx * unsigned(p.Ny) * unsigned(p.Nz) : 0u;
        t.dunits = FastDiv(nx);
        t.n1tx = (p.Nx + N1::TX - 1) / N1::TX;
        t.n1ty = (p.Ny + N1::TY - 1) / N1::TY;
        if (p.sc_on) n1columns += (long long)t.n1tx * t.n1ty;
      }
      const int slots = prepared_blocks<k_prims3_batch<real, CL, kMinB>>(kPrimX * kPrimY, CL::kSmem);
      const int n1slots = prepared_blocks<k_n1_coef_3d<S, real, N1CoefBatch<real>>>(kN1Threads, N1::kBytes);
      for (int k : order) {
        Inst& t = ti[k];
        t.nseg = prim_segments(t.p, slots, columns);
        t.n1seg = n1_segments(t.p, n1slots, n1columns);
      }
      std::stable_sort(order.begin(), order.end(), [&](int a, int c) { return ti[a].p.plane > ti[c].p.plane; });
      std::vector<SplitItem> items;
      auto group = [&](int g, auto blocks) {       // blocks(instance): blocks of its own launch, 0 for other kinds
        b.group[g] = int(items.size());
        for (int k : order) {
          const unsigned n = blocks(ti[k]);
          for (unsigned q = 0; q < n; ++q) items.push_back({k, q});
        }
        b.group[g + 1] = int(items.size());
      };
      auto over = [](unsigned n, unsigned threads) { return (n + threads - 1) / threads; };
      constexpr unsigned kMomT = sizeof(real) == 8 ? kBlock : 128;
      constexpr int kG = sizeof(real) == 8 ? 1 : 16 / int(sizeof(ST));
      group(kMoments, [&](const Inst& t) { return t.p.Nx % kG ? 0u : over(t.moments.n, kMomT); });
      group(kMomentsRagged, [&](const Inst& t) { return t.p.Nx % kG ? over(t.moments.n, kMomT) : 0u; });
      group(kPrims, [&](const Inst& t) { return unsigned(t.ncolx * t.ncoly * t.nseg); });
      auto rows = [](const Inst& t) { return unsigned(t.rowseg) * unsigned(t.p.Ny) * unsigned(t.p.Nz); };
      group(kRows, [&](const Inst& t) { return t.p.periodic_x ? rows(t) : 0u; });
      group(kRowsBounded, [&](const Inst& t) { return t.p.periodic_x ? 0u : rows(t); });
      constexpr int kPair = sizeof(real) == 8 ? 1 : 2;
      group(kNodes, [&](const Inst& t) { return t.rowseg || t.p.Nx % kPair ? 0u : over(t.nodes.n, kColThreads); });
      group(kNodesOdd, [&](const Inst& t) { return t.rowseg || t.p.Nx % kPair == 0 ? 0u : over(t.nodes.n, kColThreads); });
      group(kStrain, [&](const Inst& t) { return over(t.units, 128); });
      group(kCoef, [&](const Inst& t) { return t.p.sc_on ? unsigned(t.n1tx * t.n1ty * t.n1seg) : 0u; });
      b.ghost_blocks = unsigned(std::min((ng + 255) / 256, 4096LL));
      b.nitems = int(items.size());
      if (b.d_insts) cudaFree(b.d_insts);
      if (b.d_items) cudaFree(b.d_items);
      b.d_insts = b.d_items = nullptr;
      if (items.empty()) return LBM_OK;
      if (dev_malloc(&b.d_insts, sizeof(Inst) * ti.size()) != cudaSuccess) return LBM_ENOMEM;
      if (dev_malloc(&b.d_items, sizeof(SplitItem) * items.size()) != cudaSuccess) return LBM_ENOMEM;
      cudaMemcpy(b.d_insts, ti.data(), sizeof(Inst) * ti.size(), cudaMemcpyHostToDevice);
      cudaMemcpy(b.d_items, items.data(), sizeof(SplitItem) * items.size(), cudaMemcpyHostToDevice);
      if constexpr (sizeof(real) == 4) {
        constexpr size_t smem = RowsLayout<D, S, kHandNothing, kRowW>::kBytes;
        prepared_blocks<k_collide_rows_batch<S, false, kRowW, kRowsMinB>>(kRowW / 2, smem);
        prepared_blocks<k_collide_rows_batch<S, true, kRowW, kRowsMinB>>(kRowW / 2, smem);
      }
      return cudaGetLastError() == cudaSuccess ? LBM_OK : LBM_ECUDA;
    }

    static void enqueue(Batch& b, int parity) {
      const Inst* insts = static_cast<const Inst*>(b.d_insts);
      const SplitItem* items = static_cast<const SplitItem*>(b.d_items);
      auto launch = [&](int g, auto kern, unsigned threads, size_t smem, auto... args) {
        const int n = b.group[g + 1] - b.group[g];
        if (n == 0) return;
        launch_overlapped(kern, dim3(unsigned(n)), threads, smem, b.stream, insts, items + b.group[g], args...);
        b.launches += 1;
      };
      launch(kMoments, k_moments_batch<S, real, false>, sizeof(real) == 8 ? kBlock : 128, 0, parity);
      launch(kMomentsRagged, k_moments_batch<S, real, true>, sizeof(real) == 8 ? kBlock : 128, 0, parity);
      launch(kPrims, k_prims3_batch<real, CL, kMinB>, kPrimX * kPrimY, CL::kSmem);
      if constexpr (sizeof(real) == 4) {
        constexpr size_t smem = RowsLayout<D, S, kHandNothing, kRowW>::kBytes;
        launch(kRows, k_collide_rows_batch<S, false, kRowW, kRowsMinB>, kRowW / 2, smem, parity, b.d_errs);
        launch(kRowsBounded, k_collide_rows_batch<S, true, kRowW, kRowsMinB>, kRowW / 2, smem, parity, b.d_errs);
      }
      launch(kNodes, k_collide_batch<S, real, false, kColThreads, kColMinB>, kColThreads, 0, parity, b.d_errs);
      launch(kNodesOdd, k_collide_batch<S, real, true, kColThreads, kColMinB>, kColThreads, 0, parity, b.d_errs);
      for (int k0 = 0; b.ghost_blocks > 0 && k0 < b.n; k0 += 65535) {
        launch_overlapped(k_ghosts_batch3<S, real>, dim3(b.ghost_blocks, unsigned(std::min(b.n - k0, 65535))), 256, 0, b.stream,
                          insts + k0, parity);
        b.launches += 1;
      }
      if (!b.tuning) {
        launch(kStrain, k_n1_strain_batch3<S, real>, 128, 0);
        const int n = b.group[kCoef + 1] - b.group[kCoef];
        if (n > 0) {
          launch_overlapped(k_n1_coef_3d<S, real, N1CoefBatch<real>>, dim3(unsigned(n)), kN1Threads, N1Column<S, real>::kBytes,
                            b.stream, N1CoefBatch<real>{insts, items + b.group[kCoef]});
          b.launches += 1;
        }
      }
      enqueue_own(b, parity);
    }
  };

  using PrepFn = int (*)(Batch&);
  using EnqFn = void (*)(Batch&, int);
  template <class... T> static int batch_list(const PrepFn** pf, const EnqFn** ef) {
    static const PrepFn p[] = {&T::prepare...};
    static const EnqFn e[] = {&T::enqueue...};
    *pf = p;
    *ef = e;
    return int(sizeof...(T));
  }
  static int batch_cands(const PrepFn** pf, const EnqFn** ef) {
    if constexpr (D == 3) return batch_list<BatchSplit>(pf, ef);
    else if constexpr (sizeof(real) == 4)
      return batch_list<BatchTiles<64, 8, 2>, BatchTiles<32, 8, 4>>(pf, ef);
    else return batch_list<BatchTiles<32, 8, 1>, BatchTiles<16, 4, 4>>(pf, ef);
  }
  static int batch_ncfg() {
    const PrepFn* pf;
    const EnqFn* ef;
    return batch_cands(&pf, &ef);
  }
  static int batch_prepare(Batch& b, int cfg) {
    const PrepFn* pf;
    const EnqFn* ef;
    const int n = batch_cands(&pf, &ef);
    return pf[cfg < n ? cfg : 0](b);
  }
  static void batch_enqueue(Batch& b, int parity) {
    const PrepFn* pf;
    const EnqFn* ef;
    const int n = batch_cands(&pf, &ef);
    ef[b.tile_cfg < n ? b.tile_cfg : 0](b, parity);
  }

  static const Ops* ops() {
    static const Ops o = {&init,       &step,          &step_multipass, &macro, &autotune,
                          &batch_ncfg, &batch_prepare, &batch_enqueue,  &ntiles};
    return &o;
  }
};

}  // namespace lbm
