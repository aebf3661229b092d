// k_state.cu -- single-state kernels over an HBM-resident complex128 vector (2^n, n <= 31).
//
// Each kernel streams amplitude pairs with coalesced 16-byte loads, four pairs in flight per
// thread, 64-bit indices.  Gate arithmetic follows svqe_internal.cuh (lifting rotations,
// integer sign flips).  Reductions use a fixed grid of kRedBlocks blocks and fixed-order
// sums, so results do not depend on scheduling.
#include <algorithm>

#include "launch.h"
#include "svqe_internal.cuh"

namespace svqe {

namespace {

enum Kind { K_SWAP = 0, K_H = 1, K_ROTY = 2, K_ROTX = 3, K_ROTZ = 4, K_NEG = 5 };

__host__ __device__ inline int kind_of(int type) {
  switch (type) {
    case SV_GATE_X: case SV_GATE_CNOT: return K_SWAP;
    case SV_GATE_H: return K_H;
    case SV_GATE_RY: case SV_GATE_SINGLE_EXC: case SV_GATE_DOUBLE_EXC: return K_ROTY;
    case SV_GATE_RX: return K_ROTX;
    case SV_GATE_RZ: return K_ROTZ;
    case SV_GATE_CZ: return K_NEG;
    default: return K_SWAP;
  }
}

template <int KIND>
__device__ __forceinline__ void apply_kind(const Rot& r, double2& x, double2& y) {
  if (KIND == K_SWAP) {
    const double2 t = x; x = y; y = t;
  } else if (KIND == K_H) {
    pair_apply(SV_GATE_H, r, false, x, y);
  } else if (KIND == K_ROTY) {
    rot_apply(r, x.x, y.x);
    rot_apply(r, x.y, y.y);
  } else if (KIND == K_ROTX) {
    const Rot m = rot_inverse(r);
    rot_apply(m, x.x, y.y);
    rot_apply(r, x.y, y.x);
  } else if (KIND == K_ROTZ) {
    const Rot m = rot_inverse(r);
    rot_apply(m, x.x, x.y);
    rot_apply(r, y.x, y.y);
  }
}

template <int KIND>
__device__ __forceinline__ double grad_kind(const double2& lx, const double2& ly,
                                            const double2& px, const double2& py) {
  if (KIND == K_ROTY) return pair_grad(SV_GATE_RY, lx, ly, px, py);
  if (KIND == K_ROTX) return pair_grad(SV_GATE_RX, lx, ly, px, py);
  if (KIND == K_ROTZ) return pair_grad(SV_GATE_RZ, lx, ly, px, py);
  return 0.0;
}

constexpr int kUnroll = 4;

__global__ void k_init_basis(double2* __restrict__ psi, uint64_t N, uint64_t b) {
  const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
  for (uint64_t i = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; i < N; i += stride)
    psi[i] = make_double2(i == b ? 1.0 : 0.0, 0.0);
}

__global__ void k_prep_coefs(const DOp* __restrict__ ops, int n_ops,
                             const double* __restrict__ theta, Rot* __restrict__ coefs) {
  const int g = blockIdx.x * blockDim.x + threadIdx.x;
  if (g < n_ops) coefs[g] = make_coef(ops[g], theta).r;
}

template <int KIND>
__global__ void __launch_bounds__(kThreads, 4) k_apply(double2* __restrict__ psi, uint64_t npairs,
                                                    DOp op, const Rot* __restrict__ coef,
                                                    int inv) {
  pdl_begin();
  Rot r = *coef;
  if (inv) r = rot_inverse(r);
  const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
  for (uint64_t p0 = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; p0 < npairs;
       p0 += kUnroll * stride) {
    uint64_t ii[kUnroll];
    double2 x[kUnroll], y[kUnroll];
#pragma unroll
    for (int u = 0; u < kUnroll; ++u) {
      const uint64_t p = p0 + u * stride;
      ii[u] = insert_zeros(p, op.sb, op.k) | op.lo_or;
      if (p < npairs) {
        x[u] = psi[ii[u]];
        if (KIND != K_NEG) y[u] = psi[ii[u] ^ op.flip];
      }
    }
#pragma unroll
    for (int u = 0; u < kUnroll; ++u) {
      const uint64_t p = p0 + u * stride;
      if (p < npairs) {
        if (KIND == K_NEG) {
          psi[ii[u]] = make_double2(dneg(x[u].x), dneg(x[u].y));
        } else {
          apply_kind<KIND>(r, x[u], y[u]);
          psi[ii[u]] = x[u];
          psi[ii[u] ^ op.flip] = y[u];
        }
      }
    }
  }
}

__device__ __forceinline__ double block_sum(double v, double* red) {
  v = warp_sum(v);
  const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
  if (l == 0) red[w] = v;
  __syncthreads();
  double t = 0.0;
  if (w == 0) {
    t = (l < (int)(blockDim.x >> 5)) ? red[l] : 0.0;
    t = warp_sum(t);
  }
  return t;  // valid in thread 0
}

template <int KIND>
__global__ void __launch_bounds__(kThreads) k_adjoint(double2* __restrict__ psi,
                                                      double2* __restrict__ lam, uint64_t npairs,
                                                      DOp op, const Rot* __restrict__ coef,
                                                      double* __restrict__ partial) {
  __shared__ double red[kThreads / 32];
  pdl_begin();
  const Rot r = rot_inverse(*coef);
  const bool want = partial != nullptr;
  double acc = 0.0;
  const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
  for (uint64_t p0 = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; p0 < npairs;
       p0 += kUnroll * stride) {
    uint64_t ii[kUnroll];
    double2 px[kUnroll], py[kUnroll], lx[kUnroll], ly[kUnroll];
#pragma unroll
    for (int u = 0; u < kUnroll; ++u) {
      const uint64_t p = p0 + u * stride;
      ii[u] = insert_zeros(p, op.sb, op.k) | op.lo_or;
      if (p < npairs) {
        px[u] = psi[ii[u]];
        lx[u] = lam[ii[u]];
        if (KIND != K_NEG) {
          py[u] = psi[ii[u] ^ op.flip];
          ly[u] = lam[ii[u] ^ op.flip];
        }
      }
    }
#pragma unroll
    for (int u = 0; u < kUnroll; ++u) {
      const uint64_t p = p0 + u * stride;
      if (p < npairs) {
        if (KIND == K_NEG) {
          psi[ii[u]] = make_double2(dneg(px[u].x), dneg(px[u].y));
          lam[ii[u]] = make_double2(dneg(lx[u].x), dneg(lx[u].y));
        } else {
          if (want) acc += grad_kind<KIND>(lx[u], ly[u], px[u], py[u]);
          apply_kind<KIND>(r, px[u], py[u]);
          apply_kind<KIND>(r, lx[u], ly[u]);
          psi[ii[u]] = px[u];
          psi[ii[u] ^ op.flip] = py[u];
          lam[ii[u]] = lx[u];
          lam[ii[u] ^ op.flip] = ly[u];
        }
      }
    }
  }
  if (want) {
    const double t = block_sum(acc, red);
    if (threadIdx.x == 0) partial[blockIdx.x] = t;
  }
}

// A group as the threads of one tile read it: masks over the tile's bits, and the part of the
// table offset (or of the sign) that the tile's index decides.
struct HRec {
  uint32_t x;     // (all bits)
  uint32_t zlow;  // z mask over the tile's bits
  int32_t cls;
  int32_t pad;
  int64_t toff;   // tables: offset of the entry at tile-bit index 0
  double c;       // one term: its coefficient, the tile's sign applied
};

// acc += f v of a one-term group: the sign (-1)^popc(zu & k) as the thread's part and a mask per
// bit of u; IMAG: (i f) v = (-f v.y, f v.x).
template <int U, int UB, bool IMAG>
__device__ __forceinline__ void hpsi_term(const HRec& G, uint32_t t, uint32_t zu,
                                          const double2 (&v)[U], double2 (&acc)[U]) {
  const uint32_t s0 = (uint32_t)(__popc(t & G.zlow) & 1) << 31;
  const int chi = __double2hiint(G.c), clo = __double2loint(G.c);
#pragma unroll
  for (int u = 0; u < U; ++u) {
    uint32_t s = s0;
#pragma unroll
    for (int b = 0; b < UB; ++b)
      if ((u >> b) & 1) s ^= (zu << (31 - b)) & 0x80000000u;
    const double f = __hiloint2double(chi ^ (int)s, clo);
    if constexpr (IMAG) {
      acc[u].x = fma(dneg(f), v[u].y, acc[u].x);
      acc[u].y = fma(f, v[u].x, acc[u].y);
    } else {
      acc[u].x = fma(f, v[u].x, acc[u].x);
      acc[u].y = fma(f, v[u].y, acc[u].y);
    }
  }
}

// acc += f v of a tabulated group: the table index as the thread's part and an offset per bit
// of u.
template <int U, int TB, int UB, int CLS>
__device__ __forceinline__ void hpsi_table(const HRec& G, uint32_t t,
                                           const double2* __restrict__ tables,
                                           const double2 (&v)[U], double2 (&acc)[U]) {
  const uint32_t tl = G.zlow & ((1u << TB) - 1u), zu = G.zlow >> TB;
  const uint32_t ti0 = pext64(t, tl);
  const int sh = __popc(tl);
  uint32_t d[3];
#pragma unroll
  for (int b = 0; b < 3; ++b) d[b] = ((zu >> b) & 1u) << (sh + __popc(zu & ((1u << b) - 1u)));
  const double* tab = reinterpret_cast<const double*>(tables + G.toff);
#pragma unroll
  for (int u = 0; u < U; ++u) {
    uint32_t ti = ti0;
#pragma unroll
    for (int b = 0; b < UB; ++b)
      if ((u >> b) & 1) ti += d[b];
    if constexpr (CLS == 0) {
      const double f = tab[2 * ti];
      acc[u].x = fma(f, v[u].x, acc[u].x);
      acc[u].y = fma(f, v[u].y, acc[u].y);
    } else if constexpr (CLS == 1) {
      const double f = tab[2 * ti + 1];
      acc[u].x = fma(dneg(f), v[u].y, acc[u].x);
      acc[u].y = fma(f, v[u].x, acc[u].y);
    } else {
      group_madd(2, make_double2(tab[2 * ti], tab[2 * ti + 1]), v[u], acc[u]);
    }
  }
}

// lambda[k] = sum_g f_g(k) psi[k ^ x_g];  partial[b] = block share of Re<psi|lambda>.
//
// A block takes tiles of 256 U / S amplitudes: its threads are S slices of the group list times
// 256 / S amplitudes, U amplitudes each (k = tile base + t + u 256 / S), and the slices' sums are
// added in slice order.  S splits the groups when the state has too few amplitudes for the chip:
// at 13 qubits 32 blocks walked 100 groups one by one, 34 us.  Records are staged per tile with
// everything that only the tile's index decides, so an amplitude costs one load of psi, an
// integer op or two and two FMAs per group.  On a large state FP64 binds (2 FMA per amplitude
// and group); a software pext per amplitude and a branch on the class inside the amplitude loop
// had kept that pipe at 75 %.
template <int U, int S>
__global__ void __launch_bounds__(kThreads, U == 8 ? 2 : U == 4 ? 3 : 4) k_hpsi(
    const double2* __restrict__ psi, double2* __restrict__ lam, int n,
    const DGroup* __restrict__ groups, int n_groups, const double2* __restrict__ tables,
    double* __restrict__ partial) {
  constexpr int T = kThreads / S;
  constexpr int TB = T == 256 ? 8 : T == 128 ? 7 : T == 64 ? 6 : 5;
  constexpr int UB = U == 8 ? 3 : U == 4 ? 2 : U == 2 ? 1 : 0;
  constexpr int kStage = 128;
  __shared__ HRec sg[kStage];
  __shared__ double2 sacc[S > 1 ? kThreads * U : 1];
  __shared__ double red[kThreads / 32];
  pdl_begin();
  const int tid = threadIdx.x, slice = tid >> TB;
  const uint32_t t = tid & (T - 1);
  const uint32_t ntiles = n > TB + UB ? 1u << (n - TB - UB) : 1u;
  const uint32_t N = n >= 32 ? 0xffffffffu : 1u << n;
  double e = 0.0;
  for (uint32_t tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
    const uint32_t base = tile << (TB + UB);
    double2 acc[U];
#pragma unroll
    for (int u = 0; u < U; ++u) acc[u] = make_double2(0.0, 0.0);
    for (int g0 = 0; g0 < n_groups; g0 += kStage) {
      const int cnt = min(kStage, n_groups - g0);
      __syncthreads();
      if (tid < cnt) {
        const DGroup G = groups[g0 + tid];
        HRec h;
        h.x = (uint32_t)G.x;
        h.zlow = (uint32_t)G.zu & ((1u << (TB + UB)) - 1u);
        h.cls = G.cls;
        h.pad = 0;
        h.toff = G.toff;
        h.c = 0.0;
        const uint32_t zhi = (uint32_t)G.zu >> (TB + UB);
        if (G.cls >= 4) {
          const double2 f = tables[G.toff];
          h.c = G.cls == 4 ? f.x : f.y;
          if (__popc(tile & zhi) & 1) h.c = dneg(h.c);
        } else {
          h.toff += (int64_t)pext64(tile, zhi) << __popc(h.zlow);
        }
        sg[tid] = h;
      }
      __syncthreads();
      for (int g = slice; g < cnt; g += S) {
        const HRec& G = sg[g];
        const uint32_t kx = (base | t) ^ G.x, zu = G.zlow >> TB;
        double2 v[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
          const uint32_t k = kx ^ (uint32_t)(u << TB);
          v[u] = k < N ? psi[k] : make_double2(0.0, 0.0);
        }
        // (one loop per class: with the class tested inside the loop the FMAs of every class issue)
        switch (G.cls) {
          case 0: hpsi_table<U, TB, UB, 0>(G, t, tables, v, acc); break;
          case 1: hpsi_table<U, TB, UB, 1>(G, t, tables, v, acc); break;
          case 2: hpsi_table<U, TB, UB, 2>(G, t, tables, v, acc); break;
          case 4: hpsi_term<U, UB, false>(G, t, zu, v, acc); break;
          default: hpsi_term<U, UB, true>(G, t, zu, v, acc); break;
        }
      }
    }
    if (S > 1) {
#pragma unroll
      for (int u = 0; u < U; ++u) sacc[(slice * U + u) * T + t] = acc[u];
      __syncthreads();
      for (int i = tid; i < T * U; i += kThreads) {
        double2 a = sacc[i];
#pragma unroll
        for (int s = 1; s < S; ++s) {
          const double2 b = sacc[s * U * T + i];
          a.x += b.x;
          a.y += b.y;
        }
        const uint32_t k = base + i;  // i = u T + t
        if (k < N) {
          const double2 p = psi[k];
          e = fma(p.x, a.x, e);
          e = fma(p.y, a.y, e);
          lam[k] = a;
        }
      }
    } else {
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const uint32_t k = (base | t) + (uint32_t)(u << TB);
        if (k < N) {
          const double2 p = psi[k];
          e = fma(p.x, acc[u].x, e);
          e = fma(p.y, acc[u].y, e);
          lam[k] = acc[u];
        }
      }
    }
  }
  const double s = block_sum(e, red);
  if (threadIdx.x == 0) partial[blockIdx.x] = s;
}

// Energy only: E = <psi|H|psi> (Eq. 2), H the Pauli sum of Eq. 3 grouped by X mask:
// E = sum_g sum_k conj(psi[k]) f_g(k) psi[k ^ x_g].
// A group's operator is Hermitian (its strings carry real coefficients), so f_g(k ^ x_g) is
// the conjugate of f_g(k) and the terms at k and k ^ x_g are complex conjugates of each other:
// the sum runs over one member k of each pair (the top bit of x_g clear) and counts
// 2 Re(conj(psi[k]) f_g(k) psi[k ^ x_g]).  psi is still read once per group, with half the FP64
// work of the full lambda = H psi product: for a one-term group the sign (-1)^popc(zu & k) is
// folded into psi[k ^ x_g] by an integer op and the coefficient applied once per group and
// warp, one DFMA per amplitude.  The diagonal group (x_g = 0) takes k and k + N/2 together, each once.
// Work unit: one warp, a chunk of min(N/2, 32 kEU) consecutive pair indices of one group
// (lane l takes pair indices l, l + 32, ...), so the group record and its class are uniform.
constexpr int kEULog = 2;
constexpr int kEU = 1 << kEULog;

__device__ __forceinline__ double2 sign_flip(const double2& w, uint32_t sm) {
  return make_double2(__hiloint2double(__double2hiint(w.x) ^ sm, __double2loint(w.x)),
                      __hiloint2double(__double2hiint(w.y) ^ sm, __double2loint(w.y)));
}

__global__ void __launch_bounds__(kThreads, 4) k_expval(const double2* __restrict__ psi, int n,
                                                        const DGroup* __restrict__ groups,
                                                        int n_groups,
                                                        const double2* __restrict__ tables,
                                                        double* __restrict__ partial) {
  __shared__ double red[kThreads / 32];
  const int lane = threadIdx.x & 31;
  const int h_log = n - 1;  // N/2 pairs per group
  const int c_log = min(h_log, 5 + kEULog);
  const int upg_log = h_log - c_log;  // chunks per group (log2)
  const uint32_t C = 1u << c_log;
  const uint64_t units = (uint64_t)n_groups << upg_log;
  const uint64_t nwarps = ((uint64_t)gridDim.x * blockDim.x) >> 5;
  const uint64_t umask = (1ull << upg_log) - 1ull;
  double e = 0.0;
  uint64_t unit = ((uint64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  while (unit < units) {
    // One run of this warp's chunks of group g: the class dispatch and the coefficient are
    // taken once per run, outside the amplitude loop.
    const int g = (int)(unit >> upg_log);
    const uint64_t gend = min(units, (uint64_t)(g + 1) << upg_log);
    const DGroup G = groups[g];
    // Indices fit in 32 bits (n <= 31).
    const uint32_t xp = G.x ? (uint32_t)G.x : (1u << h_log);  // partner mask
    const uint32_t lo = (1u << (31 - __clz((int)xp))) - 1u;
    double acc = 0.0;
    // body(k, psi[k], psi[k ^ xp]) for every pair of the run; k is pair index c0 + lane + 32 u
    // with a zero bit inserted at the top bit of xp.
    auto sweep = [&](auto body) {
      for (; unit < gend; unit += nwarps) {
        const uint32_t c0 = (uint32_t)((unit & umask) << c_log);
        uint32_t k[kEU];
        double2 v[kEU], w[kEU];
#pragma unroll
        for (int u = 0; u < kEU; ++u) {
          const uint32_t t = c0 + lane + 32 * u;
          k[u] = ((t & ~lo) << 1) | (t & lo);
          if ((uint32_t)(lane + 32 * u) < C) {
            v[u] = psi[k[u]];
            w[u] = psi[k[u] ^ xp];
          } else {
            v[u] = make_double2(0.0, 0.0);
            w[u] = v[u];
          }
        }
#pragma unroll
        for (int u = 0; u < kEU; ++u) body(k[u], v[u], w[u]);
      }
    };
    double scale = 2.0;
    if (G.x == 0) {
      // Diagonal: Re f(k) |psi[k]|^2 for both members of the (k, k + N/2) pair.
      scale = 1.0;
      sweep([&](uint32_t kv, const double2& a, const double2& b) {
        double2 f1, f2;
        group_value(G, kv, tables, f1);
        group_value(G, kv ^ xp, tables, f2);
        acc = fma(f1.x, fma(a.x, a.x, a.y * a.y), acc);
        acc = fma(f2.x, fma(b.x, b.x, b.y * b.y), acc);
      });
    } else if (G.cls == 4) {
      // One term, f(k) = c (-1)^popc(zu & k) with c real: c s (v.x w.x + v.y w.y).
      scale = 2.0 * tables[G.toff].x;
      const uint32_t zu = (uint32_t)G.zu;
      sweep([&](uint32_t kv, const double2& a, const double2& b) {
        const double2 bs = sign_flip(b, (uint32_t)(__popc(kv & zu) & 1) << 31);
        acc = fma(a.x, bs.x, acc);
        acc = fma(a.y, bs.y, acc);
      });
    } else if (G.cls == 5) {
      // One term with c imaginary: Re(i c s conj(v) w) = c s (v.y w.x - v.x w.y).
      scale = 2.0 * tables[G.toff].y;
      const uint32_t zu = (uint32_t)G.zu;
      sweep([&](uint32_t kv, const double2& a, const double2& b) {
        const double2 bs = sign_flip(b, (uint32_t)(__popc(kv & zu) & 1) << 31);
        acc = fma(a.y, bs.x, acc);
        acc = fma(dneg(a.x), bs.y, acc);
      });
    } else {
      // Tabulated f(k): Re(f conj(v) w) = Re f (v.x w.x + v.y w.y) + Im f (v.y w.x - v.x w.y).
      sweep([&](uint32_t kv, const double2& a, const double2& b) {
        double2 f;
        const int cls = group_value(G, kv, tables, f);
        if (cls != 1) acc = fma(f.x, fma(a.x, b.x, a.y * b.y), acc);
        if (cls != 0) acc = fma(f.y, fma(a.y, b.x, dneg(a.x) * b.y), acc);
      });
    }
    e = fma(scale, acc, e);
  }
  const double t = block_sum(e, red);
  if (threadIdx.x == 0) partial[blockIdx.x] = t;
}

__global__ void k_sum(const double* __restrict__ partial, int count, double* __restrict__ out) {
  __shared__ double red[32];
  double v = 0.0;
  for (int i = threadIdx.x; i < count; i += blockDim.x) v += partial[i];
  const double t = block_sum(v, red);
  if (threadIdx.x == 0) out[0] = t;
}

// One warp per parameter: it finds the parameter's ops 32 at a time and adds each op's block
// shares (lane-strided, fixed order) in op order; the block after the last parameter sums the
// energy.  Scanning the op list by a whole warp replaces one thread per parameter walking it
// alone, which took 34 us for 400 parameters; only the blocks that wrote are read, so nothing
// has to be zeroed first.
__global__ void k_finish(const DOp* __restrict__ ops, int n_ops,
                         const double* __restrict__ partial, int n_params,
                         double* __restrict__ grad, const double* __restrict__ epart,
                         int n_epart, double* __restrict__ energy, double* __restrict__ theta_upd, double lr,
                         double* __restrict__ traj) {
  __shared__ double red[32];
  pdl_begin();
  if (blockIdx.x == gridDim.x - 1) {
    if (!epart) return;
    double v = 0.0;
    for (int i = threadIdx.x; i < n_epart; i += blockDim.x) v += epart[i];
    const double t = block_sum(v, red);
    if (threadIdx.x == 0) {
      energy[0] = t;
      if (traj) traj[0] = t;
    }
    return;
  }
  const int p = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, l = threadIdx.x & 31;
  if (p >= n_params) return;
  double g = 0.0;
  for (int o0 = 0; o0 < n_ops; o0 += 32) {
    unsigned hit = __ballot_sync(0xffffffffu, o0 + l < n_ops && ops[o0 + l].param == p);
    while (hit) {
      const int o = o0 + __ffs(hit) - 1;
      hit &= hit - 1u;
      const int nb = ops[o].flags;
      double v = 0.0;
      for (int b = l; b < nb; b += 32) v += partial[(size_t)o * kRedBlocks + b];
      g += warp_sum(v);
    }
  }
  if (l == 0) {
    grad[p] = g;
    if (theta_upd) theta_upd[p] = fma(-lr, g, theta_upd[p]);
  }
}

inline int grid_for(uint64_t work) {
  const uint64_t per = (uint64_t)kThreads * kUnroll;
  uint64_t g = (work + per - 1) / per;
  if (g < 1) g = 1;
  if (g > (uint64_t)kRedBlocks) g = kRedBlocks;
  return (int)g;
}

}  // namespace

cudaError_t launch_init_basis(double2* psi, int n, uint64_t b, cudaStream_t s) {
  const uint64_t N = 1ull << n;
  k_init_basis<<<grid_for(N), kThreads, 0, s>>>(psi, N, b);
  return cudaGetLastError();
}

cudaError_t launch_prep_coefs(const DOp* ops, int n_ops, const double* theta, Rot* coefs,
                              cudaStream_t s) {
  if (n_ops <= 0) return cudaSuccess;
  k_prep_coefs<<<(n_ops + 31) / 32, 32, 0, s>>>(ops, n_ops, theta, coefs);
  return cudaGetLastError();
}

cudaError_t launch_apply_op(double2* psi, int n, const DOp& op, const Rot* coef, bool inv,
                            cudaStream_t s, bool overlap) {
  const uint64_t npairs = 1ull << (n - op.k);
  const int g = grid_for(npairs);
  switch (kind_of(op.type)) {
    case K_SWAP: return launch_overlapped(k_apply<K_SWAP>, g, kThreads, 0, s, overlap, psi, npairs, op, coef, inv);
    case K_H: return launch_overlapped(k_apply<K_H>, g, kThreads, 0, s, overlap, psi, npairs, op, coef, inv);
    case K_ROTY: return launch_overlapped(k_apply<K_ROTY>, g, kThreads, 0, s, overlap, psi, npairs, op, coef, inv);
    case K_ROTX: return launch_overlapped(k_apply<K_ROTX>, g, kThreads, 0, s, overlap, psi, npairs, op, coef, inv);
    case K_ROTZ: return launch_overlapped(k_apply<K_ROTZ>, g, kThreads, 0, s, overlap, psi, npairs, op, coef, inv);
    case K_NEG: return launch_overlapped(k_apply<K_NEG>, g, kThreads, 0, s, overlap, psi, npairs, op, coef, inv);
  }
  return cudaGetLastError();
}

int adjoint_blocks(int n, const DOp& op) { return grid_for(1ull << (n - op.k)); }

cudaError_t launch_adjoint_op(double2* psi, double2* lam, int n, const DOp& op, const Rot* coef,
                              double* partial, cudaStream_t s, bool overlap) {
  const uint64_t npairs = 1ull << (n - op.k);
  const int g = grid_for(npairs);
  switch (kind_of(op.type)) {
    case K_SWAP: return launch_overlapped(k_adjoint<K_SWAP>, g, kThreads, 0, s, overlap, psi, lam, npairs, op, coef, (double*)nullptr);
    case K_H: return launch_overlapped(k_adjoint<K_H>, g, kThreads, 0, s, overlap, psi, lam, npairs, op, coef, (double*)nullptr);
    case K_ROTY: return launch_overlapped(k_adjoint<K_ROTY>, g, kThreads, 0, s, overlap, psi, lam, npairs, op, coef, partial);
    case K_ROTX: return launch_overlapped(k_adjoint<K_ROTX>, g, kThreads, 0, s, overlap, psi, lam, npairs, op, coef, partial);
    case K_ROTZ: return launch_overlapped(k_adjoint<K_ROTZ>, g, kThreads, 0, s, overlap, psi, lam, npairs, op, coef, partial);
    case K_NEG: return launch_overlapped(k_adjoint<K_NEG>, g, kThreads, 0, s, overlap, psi, lam, npairs, op, coef, (double*)nullptr);
  }
  return cudaGetLastError();
}

namespace {
// log2 of the tile of k_hpsi on n qubits: 1024 tiles or more from 15 qubits, so that the last
// round of the SMs is short.
int hpsi_tile_log(int n) { return n >= 22 ? 11 : n >= 20 ? 10 : n >= 15 ? n - 10 : 5; }
}  // namespace

int hpsi_blocks(int n) {
  const int l = hpsi_tile_log(n);
  return n <= l ? 1 : (int)std::min<uint64_t>(1ull << (n - l), kRedBlocks);
}

cudaError_t launch_hpsi(const double2* psi, double2* lam, int n, const DGroup* groups,
                        int n_groups, const double2* tables, double* partial, cudaStream_t s,
                        bool overlap) {
  const int g = hpsi_blocks(n);
#define HPSI(U, S)                                                                              \
  return launch_overlapped(k_hpsi<U, S>, g, kThreads, 0, s, overlap, psi, lam, n, groups, n_groups, \
                           tables, partial)
  switch (hpsi_tile_log(n)) {
    case 11: HPSI(8, 1);
    case 10: HPSI(4, 1);
    case 9: HPSI(2, 1);
    case 8: HPSI(2, 2);
    case 7: HPSI(2, 4);
    case 6: HPSI(2, 8);
    default: HPSI(1, 8);
  }
#undef HPSI
}

cudaError_t launch_expval(const double2* psi, int n, const DGroup* groups, int n_groups,
                          const double2* tables, double* partial, cudaStream_t s) {
  k_expval<<<kRedBlocks, kThreads, 0, s>>>(psi, n, groups, n_groups, tables, partial);
  return cudaGetLastError();
}

cudaError_t launch_sum(const double* partial, int count, double* out, cudaStream_t s) {
  k_sum<<<1, 1024, 0, s>>>(partial, count, out);
  return cudaGetLastError();
}

cudaError_t launch_finish(const DOp* ops, int n_ops, const double* partial, int n_params,
                          double* grad, const double* epart, int n_epart, double* energy,
                          double* theta_upd, double lr, double* traj, cudaStream_t s, bool overlap) {
  const int per = kThreads / 32;
  return launch_overlapped(k_finish, (n_params + per - 1) / per + 1, kThreads, 0, s, overlap, ops,
                           n_ops, partial, n_params, grad, epart, n_epart, energy, theta_upd, lr, traj);
}

}  // namespace svqe
