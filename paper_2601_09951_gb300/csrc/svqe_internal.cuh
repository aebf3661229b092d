// svqe_internal.cuh -- types and device arithmetic shared by the CUDA translation units.
//
// Design rule for GB300: FP64 issue rate is 2 DFMA/clk/SM (measured 628 G DFMA/s on the
// whole chip) against ~64 integer and ~110 FP32 lane-ops/clk/SM.  Every kernel here is
// therefore written to minimise FP64 instructions per amplitude:
//   * sign flips and multiplications by +-1, +-i are integer bit operations or swaps;
//   * the RY and RX gates of fused passes and commuting layers run without their normalisation
//     (RotT, 2 DFMA per real pair), the product of the factors left out applied once;
//   * any other real 2x2 rotation (a gate on its own, excitations) is three shears ("lifting",
//     Rot: x += a*y; y += b*x; x += a*y), 3 DFMA per real pair instead of 2 DMUL + 2 DFMA, after
//     reducing the angle to [-pi/4, pi/4] with an exact quarter-turn (a swap and sign flips);
//   * Pauli groups are applied through tabulated f_g(i), one complex or real multiply-add
//     per amplitude per group whatever the number of terms in the group.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "../../include/svqe.h"
#include "svqe_types.h"

namespace svqe {

// Negation by flipping the sign bit (an integer op: never issued to the FP64 pipe).
__device__ __forceinline__ double dneg(double v) {
  return __hiloint2double(__double2hiint(v) ^ 0x80000000, __double2loint(v));
}

// Insert zero bits at the sorted positions sb[0..k) of counter p.
__device__ __forceinline__ uint64_t insert_zeros(uint64_t p, const uint8_t* sb, int k) {
#pragma unroll
  for (int t = 0; t < 4; ++t) {
    if (t < k) {
      const uint64_t low = p & ((1ull << sb[t]) - 1ull);
      p = ((p >> sb[t]) << (sb[t] + 1)) | low;
    }
  }
  return p;
}

// Gather the bits of i selected by mask m into the low bits (software pext).
__device__ __forceinline__ uint32_t pext64(uint64_t i, uint64_t m) {
  uint32_t r = 0;
  int k = 0;
  while (m) {
    const int pos = __ffsll((long long)m) - 1;
    r |= (uint32_t)((i >> pos) & 1ull) << k;
    ++k;
    m &= m - 1;
  }
  return r;
}

// Rotation coefficients for R(phi), computed once per gate (not per amplitude).
__device__ __forceinline__ Rot make_rot_cs(double c, double s) {
  Rot r;
  double cr, sr;
  if (fabs(c) >= fabs(s)) {
    if (c >= 0) { r.k = 0; cr = c; sr = s; } else { r.k = 2; cr = -c; sr = -s; }
  } else {
    if (s > 0) { r.k = 1; cr = s; sr = -c; } else { r.k = 3; cr = -s; sr = c; }
  }
  r.a = -sr / (1.0 + cr);
  r.b = sr;
  r.pad = 0;
  return r;
}

__device__ __forceinline__ Rot make_rot(double phi) {
  double s, c;
  sincos(phi, &s, &c);
  return make_rot_cs(c, s);
}

// R(phi) without its normalisation from c = cos phi, s = sin phi: with mode 0 (|c| >= |s|)
// t = tan phi and R(phi) = f [[1, -t], [t, 1]], with mode 1 t = cot phi and
// R(phi) = f [[t, -1], [1, t]].  The factor f + flo is that of the rounded t,
// +-1 / sqrt(1 + t^2) to about 2^-100 (one Newton step from the cosine, 1 + t^2 held in two
// doubles), so that a product of factors keeps the norm of the amplitudes to one rounding.
struct RotT {
  double t, f, flo;
  int mode;
};
__device__ __forceinline__ RotT make_rott(double c, double s) {
  RotT o;
  o.mode = fabs(s) > fabs(c) ? 1 : 0;
  const double num = o.mode ? c : s, f = o.mode ? s : c;
  const double t = num / f;
  const double p = t * t, e = fma(t, t, dneg(p));
  const double a = 1.0 + p, al = (p - (a - 1.0)) + e;
  const double r2 = f * f, r2e = fma(f, f, dneg(r2));
  double res = fma(dneg(r2), a, 1.0);
  res = fma(dneg(r2e), a, res);
  res = fma(dneg(r2), al, res);
  o.t = t;
  o.f = f;
  o.flo = 0.5 * f * res;
  return o;
}
// (x, y) <- R(phi) (x, y) without the factor, or with mode 2 (from mode 1, t unchanged) or a
// negated t (mode 0) its inverse without the same factor: 2 FMA per real pair.
__device__ __forceinline__ void rot_t(int mode, double t, double& x, double& y) {
  const double u = x, v = y;
  if (mode == 0) {
    x = fma(dneg(t), v, u);
    y = fma(t, u, v);
  } else if (mode == 1) {
    x = fma(t, u, dneg(v));
    y = fma(t, v, u);
  } else {
    x = fma(t, u, v);
    y = fma(t, v, dneg(u));
  }
}
// The rotation on a pair of complex amplitudes: RY, or (ROTX) RX.
template <bool ROTX>
__device__ __forceinline__ void pair_t(int mode, double t, double2& x, double2& y) {
  if (ROTX) {
    // x' = c x - i s y, y' = c y - i s x: R(phi) on (im x, re y) and on (im y, re x)
    rot_t(mode, t, y.y, x.x);
    rot_t(mode, t, x.y, y.x);
  } else {
    rot_t(mode, t, x.x, y.x);
    rot_t(mode, t, x.y, y.y);
  }
}
// The same for RY gates without a branch on the mode.  R(phi) of mode 1 is the mode-0 form with
// its t on the swapped pair (y, x), the result for x (its inverse: for y, with -t) negated.  So
// a kernel loads the pair from swapped addresses, applies rot_y, and flips the sign of the
// amplitudes whose bit has the value `neg` when it stores them.
struct RotY {
  double t;
  uint32_t swap, neg0, neg1;  // address mask of the swap; sign masks of bit values 0 and 1
};
__device__ __forceinline__ RotY make_roty(double t, int mode, uint32_t bit, bool inv) {
  RotY r;
  r.t = inv ? dneg(t) : t;
  r.swap = mode ? bit : 0u;
  r.neg0 = mode && !inv ? 0x80000000u : 0u;
  r.neg1 = mode && inv ? 0x80000000u : 0u;
  return r;
}
__device__ __forceinline__ void rot_y(double t, double2& x, double2& y) {
  const double2 u = x, v = y;
  x.x = fma(dneg(t), v.x, u.x);
  x.y = fma(dneg(t), v.y, u.y);
  y.x = fma(t, u.x, v.x);
  y.y = fma(t, u.y, v.y);
}
__device__ __forceinline__ double2 flip_sign(const double2& v, uint32_t m) {
  return make_double2(__hiloint2double(__double2hiint(v.x) ^ (int)m, __double2loint(v.x)),
                      __hiloint2double(__double2hiint(v.y) ^ (int)m, __double2loint(v.y)));
}
// (ah + al) *= (bh + bl), both unevaluated sums, to about 2^-104.
__device__ __forceinline__ void dd_mul(double& ah, double& al, double bh, double bl) {
  const double p = ah * bh;
  double e = fma(ah, bh, dneg(p));
  e = fma(ah, bl, e);
  al = fma(al, bh, e);
  ah = p;
}

// Coefficients of R(-phi) from those of R(phi).
__device__ __forceinline__ Rot rot_inverse(const Rot& r) {
  Rot q;
  q.k = (4 - r.k) & 3;
  q.a = dneg(r.a);
  q.b = dneg(r.b);
  q.pad = 0;
  return q;
}

// (x, y) <- R(phi) (x, y): an exact quarter turn, then three shears (3 DFMA).
__device__ __forceinline__ void rot_apply(const Rot& r, double& x, double& y) {
  double u = x, v = y;
  switch (r.k) {
    case 1: u = dneg(y); v = x; break;
    case 2: u = dneg(x); v = dneg(y); break;
    case 3: u = y; v = dneg(x); break;
    default: break;
  }
  u = fma(r.a, v, u);
  v = fma(r.b, u, v);
  u = fma(r.a, v, u);
  x = u;
  y = v;
}

// ------------------------------------------------------------------------------ gate math
// Coefficients of a compiled op: rotation ops store Rot(theta/2).
struct Coef {
  Rot r;
};

__device__ __forceinline__ Coef make_coef(const DOp& op, const double* theta) {
  Coef c;
  const double t = op.param >= 0 ? theta[op.param] : op.fixed;
  if (is_param_type(op.type)) {
    c.r = make_rot(0.5 * t);
  } else {
    c.r.a = c.r.b = 0.0;
    c.r.k = 0;
    c.r.pad = 0;
  }
  return c;
}

// Apply (inv = false) or un-apply (inv = true) a pair gate to (x, y) = (psi[i], psi[j]).
__device__ __forceinline__ void pair_apply(int type, const Rot& rf, bool inv, double2& x,
                                           double2& y) {
  switch (type) {
    case SV_GATE_X:
    case SV_GATE_CNOT: {
      const double2 t = x; x = y; y = t;
    } break;
    case SV_GATE_H: {
      const double r = 0.70710678118654752440;
      const double2 a = x, b = y;
      x.x = r * (a.x + b.x); x.y = r * (a.y + b.y);
      y.x = r * (a.x - b.x); y.y = r * (a.y - b.y);
    } break;
    case SV_GATE_RY:
    case SV_GATE_SINGLE_EXC:
    case SV_GATE_DOUBLE_EXC: {
      const Rot r = inv ? rot_inverse(rf) : rf;
      rot_apply(r, x.x, y.x);
      rot_apply(r, x.y, y.y);
    } break;
    case SV_GATE_RX: {
      // x' = c x - i s y ; y' = -i s x + c y : R(-phi) on (x.re, y.im), R(phi) on (x.im, y.re)
      const Rot r = inv ? rot_inverse(rf) : rf;
      const Rot m = rot_inverse(r);
      rot_apply(m, x.x, y.y);
      rot_apply(r, x.y, y.x);
    } break;
    case SV_GATE_RZ: {
      // x *= e^{-i phi}: R(-phi) on (x.re, x.im); y *= e^{+i phi}: R(phi) on (y.re, y.im)
      const Rot r = inv ? rot_inverse(rf) : rf;
      const Rot m = rot_inverse(r);
      rot_apply(m, x.x, x.y);
      rot_apply(r, y.x, y.y);
    } break;
    default: break;
  }
}

// 2 Im<lambda|G|psi> restricted to one pair, for the generator G of a parameterised gate
// (U = exp(-i t G)): G = X/2, Y/2, Z/2 for RX/RY/RZ, sigma_y/2 on (lo, hi) for excitations.
__device__ __forceinline__ double pair_grad(int type, const double2& lx, const double2& ly,
                                            const double2& px, const double2& py) {
  switch (type) {
    case SV_GATE_RY:
    case SV_GATE_SINGLE_EXC:
    case SV_GATE_DOUBLE_EXC: {
      // Re(conj(ly) px) - Re(conj(lx) py)
      double v = ly.x * px.x;
      v = fma(ly.y, px.y, v);
      v = fma(dneg(lx.x), py.x, v);
      v = fma(dneg(lx.y), py.y, v);
      return v;
    }
    case SV_GATE_RX: {
      // Im(conj(lx) py) + Im(conj(ly) px)
      double v = lx.x * py.y;
      v = fma(dneg(lx.y), py.x, v);
      v = fma(ly.x, px.y, v);
      v = fma(dneg(ly.y), px.x, v);
      return v;
    }
    case SV_GATE_RZ: {
      // Im(conj(lx) px) - Im(conj(ly) py)
      double v = lx.x * px.y;
      v = fma(dneg(lx.y), px.x, v);
      v = fma(dneg(ly.x), py.y, v);
      v = fma(ly.y, py.x, v);
      return v;
    }
    default:
      return 0.0;
  }
}

// acc += f * v for a group table value f of class cls (0 real, 1 imaginary, 2 complex).
__device__ __forceinline__ void group_madd(int cls, const double2& f, const double2& v,
                                           double2& acc) {
  if (cls == 0) {
    acc.x = fma(f.x, v.x, acc.x);
    acc.y = fma(f.x, v.y, acc.y);
  } else if (cls == 1) {
    // (i fi) v = (-fi v.im, fi v.re)
    acc.x = fma(dneg(f.y), v.y, acc.x);
    acc.y = fma(f.y, v.x, acc.y);
  } else {
    acc.x = fma(f.x, v.x, acc.x);
    acc.x = fma(dneg(f.y), v.y, acc.x);
    acc.y = fma(f.x, v.y, acc.y);
    acc.y = fma(f.y, v.x, acc.y);
  }
}

// f_g(k) of a group (see DGroup); returns the class of the value (0 real, 1 imag, 2 complex).
__device__ __forceinline__ int group_value(const DGroup& G, uint64_t k, const double2* tables,
                                           double2& f) {
  if (G.cls >= 4) {
    f = tables[G.toff];
    if (__popcll(k & G.zu) & 1) f = make_double2(dneg(f.x), dneg(f.y));
    return G.cls - 4;
  }
  f = tables[G.toff + pext64(k, G.zu)];
  return G.cls;
}

__device__ __forceinline__ double2 cmul(const double2& a, const double2& b) {
  return make_double2(fma(a.x, b.x, dneg(a.y) * b.y), fma(a.x, b.y, a.y * b.x));
}
__device__ __forceinline__ double2 cmul_conj(const double2& a, const double2& b) {  // a conj(b)
  return make_double2(fma(a.x, b.x, a.y * b.y), fma(a.y, b.x, dneg(a.x) * b.y));
}
// acc += a conj(b)
__device__ __forceinline__ void cmac_conj(double2& acc, const double2& a, const double2& b) {
  acc.x = fma(a.x, b.x, acc.x);
  acc.x = fma(a.y, b.y, acc.x);
  acc.y = fma(a.y, b.x, acc.y);
  acc.y = fma(dneg(a.x), b.y, acc.y);
}

// Sum over the warp of 16 values per lane by recursive halving (16 DADD per lane instead of
// 80); afterwards lanes 2j and 2j+1 hold the warp total of value j.
__device__ __forceinline__ double warp_sum16(double (&v)[16]) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int s = 0; s < 4; ++s) {
    const int o = 16 >> s, h = 8 >> s;
    const bool up = (lane & o) != 0;
#pragma unroll
    for (int i = 0; i < h; ++i) {
      const double send = up ? v[i] : v[i + h];
      const double keep = up ? v[i + h] : v[i];
      v[i] = keep + __shfl_xor_sync(0xffffffffu, send, o);
    }
  }
  return v[0] + __shfl_xor_sync(0xffffffffu, v[0], 1);
}

// One-qubit gate with (cos phi, sin phi) = cs on a single qubit's state (x, y).
__device__ __forceinline__ void qubit_apply(int type, const double2& cs, double2& x, double2& y) {
  const double2 a = x, b = y;
  switch (type) {
    case SV_GATE_X: x = b; y = a; break;
    case SV_GATE_H: {
      const double r = 0.70710678118654752440;
      x = make_double2(r * (a.x + b.x), r * (a.y + b.y));
      y = make_double2(r * (a.x - b.x), r * (a.y - b.y));
    } break;
    case SV_GATE_RY:
      x = make_double2(fma(cs.x, a.x, dneg(cs.y) * b.x), fma(cs.x, a.y, dneg(cs.y) * b.y));
      y = make_double2(fma(cs.y, a.x, cs.x * b.x), fma(cs.y, a.y, cs.x * b.y));
      break;
    case SV_GATE_RX:  // x' = c x - i s y, y' = c y - i s x
      x = make_double2(fma(cs.x, a.x, cs.y * b.y), fma(cs.x, a.y, dneg(cs.y) * b.x));
      y = make_double2(fma(cs.x, b.x, cs.y * a.y), fma(cs.x, b.y, dneg(cs.y) * a.x));
      break;
    case SV_GATE_RZ:
      x = cmul_conj(a, cs);
      y = cmul(b, cs);
      break;
    default: break;
  }
}

// ------------------------------------------------------------------------------ launch overlap
// A kernel launched with launch_overlapped starts while its predecessor on the stream runs.
// Before pdl_begin it may read only what kernels before that predecessor wrote (a kernel lets
// its successor start after its own pdl_begin, so everything older is complete by then) and may
// write no global memory.
__device__ __forceinline__ void pdl_begin() {
  asm volatile("griddepcontrol.wait;" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

// ------------------------------------------------------------------------------ reductions
__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

}  // namespace svqe
