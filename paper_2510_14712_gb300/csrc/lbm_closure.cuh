// lbm_closure.cuh - the thermodynamic closures of the step: exact van der Waals
// and Peng-Robinson relations (with an FP64 temperature inversion for FP32
// arithmetic) and the learned one.
#pragma once

#include "lbm_kernels.cuh"
#include "lbm_mlp.cuh"

namespace lbm {

// Thermodynamic closures of the step: from rho, the
// specific total energy E and |u|^2 they give e = E - |u|^2/2 and
// (T, P, c_s^2).  kWarp: the closure is warp-collective (every lane calls it,
// `act` says whether the lane's node is real).  kExtra: fields the closure
// adds to the primitive ring.  kSmem: shared-memory table bytes it loads.
// kOutput: its fields are reported, not stepped with (no h, no Lambda).
// kEnergy: the collision takes e as the closure found it, not from T.
// load() runs once per CTA before the first work item.

// Exact van der Waals closure: Eqs. lbm_temp, Pvdw, vdW_speed_of_sound.
// T64 (FP32 arithmetic only): the temperature inversion of Eq. lbm_temp in
// FP64 (vdw_temperature_fp64), the mixed-precision form of the FP32 and
// FP16-deviation builds.
template <typename real, bool T64 = false> struct ExactClosure {
  static constexpr bool kPr = false;
  static constexpr bool kWarp = false, kOutput = false, kEnergy = T64 && sizeof(real) == 4;
  static constexpr int kExtra = 0;
  static constexpr size_t kSmem = 0;
  double a64 = 0.0, inv_cv64 = 0.0;
  __device__ __forceinline__ void load(const Params& p, unsigned char*) {
    if constexpr (T64) {
      a64 = p.a;
      inv_cv64 = 1.0 / p.cv;
    }
  }
  __device__ __forceinline__ void operator()(const Model<real>& m, real rho, real E, real u2, bool, real& T, real& P,
                                             real& cs2, real& e) const {
    if constexpr (T64 && sizeof(real) == 4) {
      T = vdw_temperature_fp64(a64, inv_cv64, rho, E, u2, e);
    } else {
      e = E - real(0.5) * u2;
      T = vdw_temperature(m, rho, e);
    }
    P = vdw_pressure(m, rho, T);
    cs2 = vdw_cs2(m, rho, T);
  }
};

// Exact Peng-Robinson closure: T from the quadratic in sqrt(T) of its caloric
// relation, then P and c_s^2 of the fluid, handed on to the collision with
// e = h - P/rho (kExtra = 2).  T64 (FP32 arithmetic only):
// e = E - |u|^2/2 and the root's argument e - B0 in FP64, rounded once; the
// root itself has only positive terms and stays in FP32.
template <typename real, bool T64 = false> struct PrClosure {
  static constexpr bool kPr = true;
  static constexpr bool kWarp = false, kOutput = false, kEnergy = false;
  static constexpr int kExtra = 2;
  static constexpr size_t kSmem = 0;
  __device__ __forceinline__ void load(const Params&, unsigned char*) {}
  __device__ __forceinline__ void operator()(const Model<real>& m, real rho, real E, real u2, bool, real& T, real& P,
                                             real& cs2, real& e) const {
    if constexpr (T64 && sizeof(real) == 4) {
      const double ed = double(E) - 0.5 * double(u2);
      e = real(ed);
      T = pr_temperature_q(m, rho, ed);
    } else {
      e = E - real(0.5) * u2;
      T = pr_temperature(m, rho, e);
    }
    P = pr_pressure(m, rho, T);
    cs2 = pr_cs2(m, rho, T);
  }
};

// The exact closure of the handle's fluid and temperature form, chosen at run
// time (Model::kind, Params::t64): the fields that lbm_moments reports and the
// multi-pass step.
template <typename real> struct AnyClosure {
  static constexpr bool kWarp = false, kOutput = true, kEnergy = false;
  static constexpr int kExtra = 0;
  static constexpr size_t kSmem = 0;
  ExactClosure<real, true> vdw64;
  bool t64;
  __device__ __forceinline__ void load(const Params& p, unsigned char* smem) {
    vdw64.load(p, smem);
    t64 = sizeof(real) == 4 && p.t64;
  }
  __device__ __forceinline__ void operator()(const Model<real>& m, real rho, real E, real u2, bool act, real& T,
                                             real& P, real& cs2, real& e) const {
    if (m.kind == LBM_EOS_PR) {
      if (t64) PrClosure<real, true>()(m, rho, E, u2, act, T, P, cs2, e);
      else PrClosure<real>()(m, rho, E, u2, act, T, P, cs2, e);
    } else if (t64) {
      vdw64(m, rho, E, u2, act, T, P, cs2, e);
    } else {
      ExactClosure<real>()(m, rho, E, u2, act, T, P, cs2, e);
    }
  }
};

// Learned closure: the network of lbm_mlp.cuh inside its training box, the
// exact closure outside it (range gate).  FP32 arithmetic only.
struct MlpClosure {
  static constexpr bool kPr = false;
  static constexpr bool kWarp = true, kOutput = false, kEnergy = false;
  static constexpr int kExtra = 2;
  static constexpr size_t kSmem = sizeof(mlp::Image);
  const mlp::Image* w;
  __device__ __forceinline__ void load(const Params& p, unsigned char* smem) {
    mlp::Image* d = reinterpret_cast<mlp::Image*>(smem);
    mlp::load_image(static_cast<const mlp::Image*>(p.mlp), d);
    w = d;
  }
  __device__ __forceinline__ void operator()(const Model<float>& m, float rho, float E, float u2, bool act, float& T,
                                             float& P, float& cs2, float& e) const {
    e = E - 0.5f * u2;
    mlp::closure_warp(*w, m, rho, e, act, T, P, cs2);
  }
};

// v mod n in [0, n) for any integer v
__device__ __forceinline__ int modp(int v, int n) {
  const int r = v % n;
  return r < 0 ? r + n : r;
}

}  // namespace lbm
