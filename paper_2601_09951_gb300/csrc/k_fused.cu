// k_fused.cu -- fused passes of the single-state path (see FPass): a tile of 2^m amplitudes
// is staged in shared memory, a whole run of gates is applied to it, and it is written back,
// so the run costs one read and one write of the HBM-resident state instead of one per gate.
//
// Forward:  k_fpass applies the pass's items to psi.
// Backward: k_bpass stages psi and lambda, walks the items in reverse, accumulates each
//           parameterised item's 2 Im<lambda|G|psi> in a per-thread shared-memory slot (one
//           DADD per item per tile instead of a warp reduction), un-applies the items to both,
//           and reduces every slot once at the end into partial[op * kRedBlocks + block] (one
//           block per tile up to kRedBlocks).
// A run of RZ gates is one diagonal phase per amplitude: half tables over the tile's local
// bits times a per-tile factor for the RZ gates on outer bits.
//
// What bounds these kernels is the FP64 pipe (2 FMA/clk/SM), so the RY and RX gates of a pass
// run without their normalisation: R(phi) = cos phi [[1, -t], [t, 1]] with t = tan phi is two
// FMAs per real pair where three shears are three, and the product of the cosines multiplies
// the tile once, when it is stored (SItem; cot and sin where |sin| > |cos|, so every factor
// dropped lies in [0.707, 1]).  Two such gates on different bits share one trip through shared
// memory.  The pass's items, coefficients included, are staged in shared memory by one warp while
// the tile's loads are in flight: read one at a time from global memory they cost a round trip
// per gate and tile, which is most of a pass when a state of 2^13 to 2^20 amplitudes sits in L2.
// Nothing is computed per item here: one warp's FP64 instruction takes 64 clocks of its
// scheduler's pipe, so a chain of 40 of them costs a block 1.2 us, once per block of every pass
// (k_prep.cu does it once per evaluation).
#include <algorithm>

#include "launch.h"
#include "svqe_internal.cuh"

namespace svqe {

namespace {

constexpr int kFT = 256;  // threads per CTA of the fused kernels

struct DiagS {
  double2 cs[kMaxSlotsDev];  // (cos phi, sin phi) per RZ gate of the item
  int loc[kMaxSlotsDev];     // local bit, or -1 - global bit for a gate on an outer bit
  int par[kMaxSlotsDev];     // whether the gate has a gradient
  double2 tl[64];            // phase over local bits [0, hl)
  double2 th[64];            // phase over local bits [hl, m), times the tile's outer factor
  double2 th0[64];           // phase over local bits [hl, m) alone
  int m_rz;
  int hl;
};

__device__ __forceinline__ double2 rz_factor(const double2& cs, int bit) {
  return make_double2(cs.x, bit ? cs.y : dneg(cs.y));  // e^{-i phi} on |0>, e^{+i phi} on |1>
}

__device__ __forceinline__ uint32_t pdep32(uint32_t v, uint32_t m) {
  uint32_t r = 0;
  while (m) {
    const uint32_t low = m & (0u - m);
    if (v & 1u) r |= low;
    v >>= 1;
    m &= m - 1u;
  }
  return r;
}

// Per-CTA setup of a diagonal item: cos/sin, local bits and the inner half tables.
__device__ void diag_setup(DiagS& D, const FPass& P, int op0, int count, const DOp* gops,
                           const double2* cs) {
  if (threadIdx.x == 0) {
    D.m_rz = count;
    D.hl = P.m / 2;
  }
  if ((int)threadIdx.x < count) {
    D.cs[threadIdx.x] = cs[op0 + threadIdx.x];
    const int bit0 = gops[op0 + threadIdx.x].bit0;
    const uint64_t b = 1ull << bit0;
    D.loc[threadIdx.x] = (P.tile_mask & b) ? __popcll(P.tile_mask & (b - 1ull)) : -1 - bit0;
    D.par[threadIdx.x] = gops[op0 + threadIdx.x].param >= 0;
  }
  __syncthreads();
  const int hl = D.hl;
  const int nl = 1 << hl, nh = 1 << (P.m - hl);
  for (int j = threadIdx.x; j < nl + nh; j += blockDim.x) {
    const bool hi = j >= nl;
    const int jj = hi ? j - nl : j;
    double2 p = make_double2(1.0, 0.0);
    for (int g = 0; g < D.m_rz; ++g) {
      const int lb = D.loc[g];
      if (lb < 0 || (lb >= hl) != hi) continue;
      p = cmul(p, rz_factor(D.cs[g], (jj >> (hi ? lb - hl : lb)) & 1));
    }
    if (hi) D.th0[jj] = p; else D.tl[jj] = p;
  }
  __syncthreads();
}

// Per-tile: th = th0 * (product of the outer-bit RZ factors for this tile), the product by a
// tree over the lanes of each warp that needs it.
__device__ void diag_tile(DiagS& D, const FPass& P, uint32_t outer) {
  const int nh = 1 << (P.m - D.hl), lane = threadIdx.x & 31;
  if ((int)(threadIdx.x & ~31u) >= nh) return;
  double2 f = make_double2(1.0, 0.0);
  if (lane < D.m_rz && D.loc[lane] < 0)
    f = rz_factor(D.cs[lane], (int)((outer >> (-1 - D.loc[lane])) & 1u));
#pragma unroll
  for (int o = 8; o > 0; o >>= 1) {
    const double x = __shfl_xor_sync(0xffffffffu, f.x, o), y = __shfl_xor_sync(0xffffffffu, f.y, o);
    f = cmul(f, make_double2(x, y));
  }
  f.x = __shfl_sync(0xffffffffu, f.x, 0);
  f.y = __shfl_sync(0xffffffffu, f.y, 0);
  for (int j = threadIdx.x; j < nh; j += blockDim.x) D.th[j] = cmul(D.th0[j], f);
}

__device__ __forceinline__ double2 diag_phase(const DiagS& D, uint32_t j) {
  return cmul(D.th[j >> D.hl], D.tl[j & ((1u << D.hl) - 1u)]);
}

// Asynchronous 16-byte global -> shared copies (cp.async, L2 only): a tile's loads are all in
// flight at once instead of one round trip per loop iteration; cp_async_wait_all and a
// barrier complete them.
__device__ __forceinline__ void cp_async16(void* smem, const void* gmem) {
  const uint32_t d = (uint32_t)__cvta_generic_to_shared(smem);
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(d), "l"(gmem) : "memory");
}
__device__ __forceinline__ void cp_async_wait_all() {
  asm volatile("cp.async.wait_all;" ::: "memory");
}

// A thread's amplitudes of a tile are j = tid + i nt, i < 2^m / nt (nt threads, a power of
// two): the global index of j is g ^ the bits of i, g the spread of tid over the tile's bits and
// h[q] the global bit of local bit log2(nt) + q.
struct TileMap {
  uint32_t g, h[3];
  int cnt;  // amplitudes per thread (at most 8); 0 for a thread beyond the tile
};

__device__ __forceinline__ TileMap tile_map(const FPass& P) {
  TileMap T;
  const int lt = 31 - __clz((int)blockDim.x);
  uint32_t m = (uint32_t)P.tile_mask, v = threadIdx.x;
  T.g = 0;
  for (int b = 0; b < lt && m; ++b) {
    const uint32_t low = m & (0u - m);
    if (v & 1u) T.g |= low;
    v >>= 1;
    m &= m - 1u;
  }
#pragma unroll
  for (int q = 0; q < 3; ++q) {
    T.h[q] = m & (0u - m);
    m &= m - 1u;
  }
  T.cnt = P.m > lt ? 1 << (P.m - lt) : (threadIdx.x < (1u << P.m) ? 1 : 0);
  return T;
}
__device__ __forceinline__ uint32_t tile_idx(const TileMap& T, int i) {
  return T.g ^ ((i & 1) ? T.h[0] : 0u) ^ ((i & 2) ? T.h[1] : 0u) ^ ((i & 4) ? T.h[2] : 0u);
}

constexpr int kChunk = 32;  // items staged at a time, one lane of the first warp each

// Stage items [0, cnt) of the chunk at src (cnt <= kChunk) by the first warp, inverted for
// un-applying: the inverse of (p x - y, x + p y) is (p x + y, p y - x) with the same factor left
// out.
__device__ __forceinline__ void stage_items(SItem* S, const SItem* src, int cnt, bool inv) {
  const int lane = threadIdx.x;
  if (lane >= cnt) return;
  SItem o = src[lane];
  if (inv) {
    if (o.kind == F_RY || o.kind == F_RX) {
      if (o.mode) o.mode = 2;
      else o.p = dneg(o.p);
    } else if (o.kind == F_EXC || o.kind == F_ROTZ) {
      o.p = dneg(o.p);
      o.q = dneg(o.q);
      o.mode = (int16_t)((4 - o.mode) & 3);
    }
  }
  S[lane] = o;
}

// Which of the thread's amplitudes (bit i: j = tid + i nt) some item of a sparse pass touches: the
// others are neither read nor written (see FPass::sparse).
__device__ __forceinline__ uint32_t touched(const SItem* its, int n_items, const TileMap& T) {
  uint32_t need = 0;
  for (int q = 0; q < n_items; ++q) {
    const SItem& s = its[q];
    uint32_t wires = 0;
#pragma unroll
    for (int t = 0; t < 4; ++t)
      if (t < s.k) wires |= 1u << s.sb[t];
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const uint32_t w = (threadIdx.x + i * blockDim.x) & wires;
      if (i < T.cnt && (w == s.lo || w == (s.lo ^ s.fl))) need |= 1u << i;
    }
  }
  return need;
}

// One pair of one of the normalised kinds.
template <int KIND>
__device__ __forceinline__ void fapply(const SItem& s, double2& x, double2& y) {
  if (KIND == F_SWAP) {
    const double2 t = x; x = y; y = t;
  } else if (KIND == F_H) {
    pair_apply(SV_GATE_H, Rot{}, false, x, y);
  } else if (KIND == F_EXC) {
    const Rot r{s.p, s.q, s.mode, 0};
    rot_apply(r, x.x, y.x);
    rot_apply(r, x.y, y.y);
  } else if (KIND == F_ROTZ) {
    const Rot r{s.p, s.q, s.mode, 0};
    const Rot m = rot_inverse(r);
    rot_apply(m, x.x, x.y);
    rot_apply(r, y.x, y.y);
  } else if (KIND == F_RY) {
    pair_t<false>(s.mode, s.p, x, y);
  } else if (KIND == F_RX) {
    pair_t<true>(s.mode, s.p, x, y);
  }
}

// acc += 2 Im<lambda|G|psi> on one pair, folded into FMAs.
template <int KIND>
__device__ __forceinline__ void fgrad(const double2& lx, const double2& ly, const double2& px,
                                      const double2& py, double& acc) {
  if (KIND == F_RX) {
    acc = fma(lx.x, py.y, acc);
    acc = fma(dneg(lx.y), py.x, acc);
    acc = fma(ly.x, px.y, acc);
    acc = fma(dneg(ly.y), px.x, acc);
  } else if (KIND == F_ROTZ) {
    acc = fma(lx.x, px.y, acc);
    acc = fma(dneg(lx.y), px.x, acc);
    acc = fma(dneg(ly.x), py.y, acc);
    acc = fma(ly.y, py.x, acc);
  } else if (KIND == F_RY || KIND == F_EXC) {
    acc = fma(ly.x, px.x, acc);
    acc = fma(ly.y, px.y, acc);
    acc = fma(dneg(lx.x), py.x, acc);
    acc = fma(dneg(lx.y), py.y, acc);
  }
}

__device__ __forceinline__ uint32_t item_index(const SItem& s, uint32_t p) {
#pragma unroll
  for (int t = 0; t < 4; ++t) {
    if (t < s.k) {
      const uint32_t low = p & ((1u << s.sb[t]) - 1u);
      p = ((p >> s.sb[t]) << (s.sb[t] + 1)) | low;
    }
  }
  return p | s.lo;
}

template <int KIND>
__device__ __forceinline__ void tile_op_k(double2* v, uint32_t M, const SItem& s) {
  const uint32_t np = M >> s.k, nt = blockDim.x;
  for (uint32_t p = threadIdx.x; p < np; p += nt) {
    const uint32_t i = item_index(s, p);
    if (KIND == F_NEG) {
      v[i] = make_double2(dneg(v[i].x), dneg(v[i].y));
    } else {
      double2 x = v[i], y = v[i ^ s.fl];
      fapply<KIND>(s, x, y);
      v[i] = x;
      v[i ^ s.fl] = y;
    }
  }
}

__device__ __forceinline__ void tile_op(double2* v, uint32_t M, const SItem& s) {
  switch (s.kind) {
    case F_SWAP: tile_op_k<F_SWAP>(v, M, s); break;
    case F_H: tile_op_k<F_H>(v, M, s); break;
    case F_EXC: tile_op_k<F_EXC>(v, M, s); break;
    case F_ROTZ: tile_op_k<F_ROTZ>(v, M, s); break;
    case F_RY: tile_op_k<F_RY>(v, M, s); break;
    case F_RX: tile_op_k<F_RX>(v, M, s); break;
    default: tile_op_k<F_NEG>(v, M, s); break;
  }
}

// The four amplitudes of a block on two single-bit items: i, i | f0, i | f1, i | f0 | f1.
__device__ __forceinline__ uint32_t quad_index(uint32_t f0, uint32_t f1, uint32_t p) {
  const uint32_t l0 = min(f0, f1) - 1u, l1 = max(f0, f1) - 1u;
  p = ((p & ~l0) << 1) | (p & l0);
  return ((p & ~l1) << 1) | (p & l1);
}

// Two RY (or RX) gates on different bits in one trip, s0 first.
template <bool ROTX>
__device__ __forceinline__ void tile_op2(double2* v, uint32_t M, const SItem& s0,
                                         const SItem& s1) {
  const uint32_t f0 = s0.fl, f1 = s1.fl, nt = blockDim.x;
  const int m0 = s0.mode, m1 = s1.mode;
  const double t0 = s0.p, t1 = s1.p;
  for (uint32_t p = threadIdx.x; p < (M >> 2); p += nt) {
    const uint32_t i = quad_index(f0, f1, p);
    double2 a = v[i], b = v[i | f0], c = v[i | f1], d = v[i | f0 | f1];
    pair_t<ROTX>(m0, t0, a, b);
    pair_t<ROTX>(m0, t0, c, d);
    pair_t<ROTX>(m1, t1, a, c);
    pair_t<ROTX>(m1, t1, b, d);
    v[i] = a;
    v[i | f0] = b;
    v[i | f1] = c;
    v[i | f0 | f1] = d;
  }
}

// Adjoint step of one item on the psi and lambda tiles: gradient share into acc, then un-apply
// to both.
template <int KIND>
__device__ __forceinline__ void tile_adj_k(double2* tp, double2* tl, uint32_t M, const SItem& s,
                                           double& acc) {
  const uint32_t np = M >> s.k, nt = blockDim.x;
  const bool grad = s.slot >= 0;
  for (uint32_t p = threadIdx.x; p < np; p += nt) {
    const uint32_t a = item_index(s, p);
    if (KIND == F_NEG) {
      tp[a] = make_double2(dneg(tp[a].x), dneg(tp[a].y));
      tl[a] = make_double2(dneg(tl[a].x), dneg(tl[a].y));
    } else {
      const uint32_t b = a ^ s.fl;
      double2 px = tp[a], py = tp[b], lx = tl[a], ly = tl[b];
      if (grad) fgrad<KIND>(lx, ly, px, py, acc);
      fapply<KIND>(s, px, py);
      fapply<KIND>(s, lx, ly);
      tp[a] = px;
      tp[b] = py;
      tl[a] = lx;
      tl[b] = ly;
    }
  }
}

// The same for one RY or RX gate (a pass's odd one), compiled per mode: with the mode chosen inside
// the loop a gate of mode 2 issued the FP64 work of both (24 qubits, 7 and 11 gates: 1388 and
// 2064 us with such a gate, 1250 and 1930 now with either mode).
template <int KIND, int MODE>
__device__ __forceinline__ void tile_adj_rot(double2* tp, double2* tl, uint32_t M, const SItem& s,
                                             double& acc) {
  constexpr bool ROTX = KIND == F_RX;
  const uint32_t np = M >> 1, nt = blockDim.x;
  const bool grad = s.slot >= 0;
  const uint32_t fl = s.fl;
  const double t = s.p;
  for (uint32_t p = threadIdx.x; p < np; p += nt) {
    const uint32_t low = p & (fl - 1u), a = ((p ^ low) << 1) | low, b = a | fl;
    double2 px = tp[a], py = tp[b], lx = tl[a], ly = tl[b];
    if (grad) fgrad<KIND>(lx, ly, px, py, acc);
    pair_t<ROTX>(MODE, t, px, py);
    pair_t<ROTX>(MODE, t, lx, ly);
    tp[a] = px;
    tp[b] = py;
    tl[a] = lx;
    tl[b] = ly;
  }
}
template <int KIND>
__device__ __forceinline__ void tile_adj_rot(double2* tp, double2* tl, uint32_t M, const SItem& s,
                                             double& acc) {
  if (s.mode == 0) tile_adj_rot<KIND, 0>(tp, tl, M, s, acc);
  else tile_adj_rot<KIND, 2>(tp, tl, M, s, acc);  // (an inverse has no mode 1)
}

// The same for two RY (or RX) gates on different bits, s0 un-applied first.
template <bool ROTX>
__device__ __forceinline__ void tile_adj2(double2* tp, double2* tl, uint32_t M, const SItem& s0,
                                          const SItem& s1, double& acc0, double& acc1) {
  constexpr int KIND = ROTX ? F_RX : F_RY;
  const uint32_t f0 = s0.fl, f1 = s1.fl, nt = blockDim.x;
  const int m0 = s0.mode, m1 = s1.mode;
  const double t0 = s0.p, t1 = s1.p;
  const bool g0 = s0.slot >= 0, g1 = s1.slot >= 0;
  for (uint32_t p = threadIdx.x; p < (M >> 2); p += nt) {
    const uint32_t i = quad_index(f0, f1, p), j = i | f0, k = i | f1, l = j | f1;
    double2 pa = tp[i], pb = tp[j], pc = tp[k], pd = tp[l];
    double2 la = tl[i], lb = tl[j], lc = tl[k], ld = tl[l];
    if (g0) {
      fgrad<KIND>(la, lb, pa, pb, acc0);
      fgrad<KIND>(lc, ld, pc, pd, acc0);
    }
    pair_t<ROTX>(m0, t0, pa, pb);
    pair_t<ROTX>(m0, t0, pc, pd);
    pair_t<ROTX>(m0, t0, la, lb);
    pair_t<ROTX>(m0, t0, lc, ld);
    if (g1) {
      fgrad<KIND>(la, lc, pa, pc, acc1);
      fgrad<KIND>(lb, ld, pb, pd, acc1);
    }
    pair_t<ROTX>(m1, t1, pa, pc);
    pair_t<ROTX>(m1, t1, pb, pd);
    pair_t<ROTX>(m1, t1, la, lc);
    pair_t<ROTX>(m1, t1, lb, ld);
    tp[i] = pa;
    tp[j] = pb;
    tp[k] = pc;
    tp[l] = pd;
    tl[i] = la;
    tl[j] = lb;
    tl[k] = lc;
    tl[l] = ld;
  }
}

// Whether items a and b (in processing order) share a trip.
__device__ __forceinline__ bool can_pair(const SItem& a, const SItem& b) {
  return a.kind == b.kind && (a.kind == F_RY || a.kind == F_RX) && a.fl != b.fl;
}

// INV: apply the pass's items inverted, in reverse order (un-applying the pass).
template <bool INV>
__global__ void __launch_bounds__(kFT, 4) k_fpass(double2* __restrict__ psi, FPass P,
                                               const SItem* __restrict__ items,
                                               const DOp* __restrict__ gops,
                                               const double2* __restrict__ cs,
                                               const double* __restrict__ scale) {
  extern __shared__ double2 tile[];
  __shared__ DiagS D;
  __shared__ SItem its[kChunk];
  const uint32_t M = 1u << P.m, nt = blockDim.x;
  const uint64_t ntiles = 1ull << __popcll(P.outer_mask);
  const int nch = (P.n_items + kChunk - 1) / kChunk;
  const TileMap T = tile_map(P);
  const double f = *scale;
  items += P.first_item;
  if (nch == 1 && threadIdx.x < 32) stage_items(its, items, P.n_items, INV);
  if (P.diag >= 0) diag_setup(D, P, items[P.diag].op, items[P.diag].count, gops, cs);
  uint32_t need = (1u << T.cnt) - 1u;
  if (P.sparse && nch == 1) {
    __syncthreads();
    need = touched(its, P.n_items, T);
  }
  pdl_begin();
  for (uint64_t t = blockIdx.x; t < ntiles; t += gridDim.x) {
    const uint32_t outer = pdep32((uint32_t)t, (uint32_t)P.outer_mask);
#pragma unroll
    for (int i = 0; i < 8; ++i)
      if ((need >> i) & 1u)
        cp_async16(&tile[threadIdx.x + i * nt], &psi[outer | tile_idx(T, i)]);
    if (P.diag >= 0) diag_tile(D, P, outer);
    for (int ch = 0; ch < nch; ++ch) {
      const int base = (INV ? nch - 1 - ch : ch) * kChunk;
      const int cnt = min(kChunk, P.n_items - base);
      if (nch > 1 && threadIdx.x < 32) stage_items(its, items + base, cnt, INV);
      if (ch == 0) cp_async_wait_all();
      __syncthreads();
      for (int ii = 0; ii < cnt;) {
        const int i = INV ? cnt - 1 - ii : ii;
        const SItem& s = its[i];
        if (s.kind == F_DIAG) {
          if (INV) {
            for (uint32_t j = threadIdx.x; j < M; j += nt)
              tile[j] = cmul_conj(tile[j], diag_phase(D, j));
          } else {
            for (uint32_t j = threadIdx.x; j < M; j += nt)
              tile[j] = cmul(tile[j], diag_phase(D, j));
          }
          ++ii;
        } else if (ii + 1 < cnt && can_pair(s, its[INV ? i - 1 : i + 1])) {
          const SItem& s1 = its[INV ? i - 1 : i + 1];
          if (s.kind == F_RX) tile_op2<true>(tile, M, s, s1);
          else tile_op2<false>(tile, M, s, s1);
          ii += 2;
        } else {
          tile_op(tile, M, s);
          ++ii;
        }
        __syncthreads();
      }
    }
    // (two loops: a select would issue the multiplications of an unscaled pass too)
    if (f == 1.0) {
#pragma unroll
      for (int i = 0; i < 8; ++i)
        if ((need >> i) & 1u) psi[outer | tile_idx(T, i)] = tile[threadIdx.x + i * nt];
    } else {
#pragma unroll
      for (int i = 0; i < 8; ++i)
        if (i < T.cnt) {
          const double2 v = tile[threadIdx.x + i * nt];
          psi[outer | tile_idx(T, i)] = make_double2(f * v.x, f * v.y);
        }
    }
    __syncthreads();
  }
}

__global__ void __launch_bounds__(kFT, 2) k_bpass(double2* __restrict__ psi,
                                               double2* __restrict__ lam, FPass P,
                                               const SItem* __restrict__ items,
                                               const DOp* __restrict__ gops,
                                               const double2* __restrict__ cs,
                                               const double* __restrict__ scale,
                                               double* __restrict__ partial) {
  extern __shared__ double2 smem[];
  __shared__ DiagS D;
  __shared__ SItem its[kChunk];
  __shared__ int s_op[kMaxSlotsDev];      // op and gradient factor of each slot
  __shared__ double s_fac[kMaxSlotsDev];
  const uint32_t M = 1u << P.m, nt = blockDim.x;
  double2* tp = smem;
  double2* tlam = smem + M;
  double* accp = (double*)(smem + 2 * M);  // [n_slots][nt]
  const uint64_t ntiles = 1ull << __popcll(P.outer_mask);
  const int tid = threadIdx.x, lt = 31 - __clz((int)nt);
  const int nch = (P.n_items + kChunk - 1) / kChunk;
  const TileMap T = tile_map(P);
  const double f = *scale;
  items += P.first_item;
  for (int s = 0; s < P.n_slots; ++s) accp[s * nt + tid] = 0.0;
  if (nch == 1 && tid < 32) stage_items(its, items, P.n_items, true);
  // op and gradient factor of each slot
  for (int i = tid; i < P.n_items; i += nt) {
    const int slot = items[i].slot;
    if (slot >= 0 && items[i].kind != F_DIAG) {
      s_op[slot] = items[i].op;
      s_fac[slot] = items[i].f;
    }
  }
  if (P.diag >= 0) {
    diag_setup(D, P, items[P.diag].op, items[P.diag].count, gops, cs);
    if (tid == 0) {
      int sl = items[P.diag].slot;
      for (int g = 0; g < D.m_rz; ++g) {
        if (!D.par[g]) continue;
        s_op[sl] = items[P.diag].op + g;
        s_fac[sl++] = items[P.diag].f;
      }
    }
  }
  uint32_t need = (1u << T.cnt) - 1u;
  if (P.sparse && nch == 1) {
    __syncthreads();
    need = touched(its, P.n_items, T);
  }
  pdl_begin();
  for (uint64_t t = blockIdx.x; t < ntiles; t += gridDim.x) {
    const uint32_t outer = pdep32((uint32_t)t, (uint32_t)P.outer_mask);
#pragma unroll
    for (int i = 0; i < 8; ++i)
      if ((need >> i) & 1u) {
        const uint32_t k = outer | tile_idx(T, i);
        cp_async16(&tp[tid + i * nt], &psi[k]);
        cp_async16(&tlam[tid + i * nt], &lam[k]);
      }
    if (P.diag >= 0) diag_tile(D, P, outer);
    for (int ch = nch - 1; ch >= 0; --ch) {
      const int base = ch * kChunk;
      const int cnt = min(kChunk, P.n_items - base);
      if (nch > 1 && tid < 32) stage_items(its, items + base, cnt, true);
      if (ch == nch - 1) cp_async_wait_all();
      __syncthreads();
      for (int i = cnt - 1; i >= 0;) {
        const SItem& s = its[i];
        if (s.kind == F_DIAG) {
          // gradients of the RZ gates: 2 Im<lambda|Z_q/2|psi> = sum_k s_q(k) Im(conj(l_k) p_k)
          double W = 0.0;
          double hi[3] = {0.0, 0.0, 0.0};  // RZ gates on local bits that vary within a thread
          for (uint32_t j = tid; j < M; j += nt) {
            const double2 pk = tp[j], lk = tlam[j];
            const double w = fma(lk.x, pk.y, dneg(lk.y) * pk.x);
            W += w;
#pragma unroll
            for (int q = 0; q < 3; ++q) hi[q] += ((j >> (lt + q)) & 1u) ? dneg(w) : w;
            const double2 ph = diag_phase(D, j);
            tp[j] = cmul_conj(pk, ph);
            tlam[j] = cmul_conj(lk, ph);
          }
          int sl = s.slot;
          for (int g = 0; g < s.count; ++g) {
            if (!D.par[g]) continue;
            const int lb = D.loc[g];
            double v;
            if (lb < 0) {
              v = ((outer >> (-1 - lb)) & 1u) ? dneg(W) : W;
            } else if (lb < lt) {
              v = ((tid >> lb) & 1) ? dneg(W) : W;
            } else {
              v = lb == lt ? hi[0] : lb == lt + 1 ? hi[1] : hi[2];
            }
            accp[sl * nt + tid] += v;
            ++sl;
          }
          --i;
        } else if (i > 0 && can_pair(s, its[i - 1])) {
          const SItem& s1 = its[i - 1];
          double a0 = 0.0, a1 = 0.0;
          if (s.kind == F_RX) tile_adj2<true>(tp, tlam, M, s, s1, a0, a1);
          else tile_adj2<false>(tp, tlam, M, s, s1, a0, a1);
          if (s.slot >= 0) accp[s.slot * nt + tid] += a0;
          if (s1.slot >= 0) accp[s1.slot * nt + tid] += a1;
          i -= 2;
        } else {
          double acc = 0.0;
          switch (s.kind) {
            case F_SWAP: tile_adj_k<F_SWAP>(tp, tlam, M, s, acc); break;
            case F_H: tile_adj_k<F_H>(tp, tlam, M, s, acc); break;
            case F_EXC: tile_adj_k<F_EXC>(tp, tlam, M, s, acc); break;
            case F_ROTZ: tile_adj_k<F_ROTZ>(tp, tlam, M, s, acc); break;
            case F_RY: tile_adj_rot<F_RY>(tp, tlam, M, s, acc); break;
            case F_RX: tile_adj_rot<F_RX>(tp, tlam, M, s, acc); break;
            default: tile_adj_k<F_NEG>(tp, tlam, M, s, acc); break;
          }
          if (s.slot >= 0) accp[s.slot * nt + tid] += acc;
          --i;
        }
        __syncthreads();
      }
    }
    if (f == 1.0) {
#pragma unroll
      for (int i = 0; i < 8; ++i)
        if ((need >> i) & 1u) {
          const uint32_t k = outer | tile_idx(T, i);
          psi[k] = tp[tid + i * nt];
          lam[k] = tlam[tid + i * nt];
        }
    } else {
#pragma unroll
      for (int i = 0; i < 8; ++i)
        if (i < T.cnt) {
          const uint32_t k = outer | tile_idx(T, i);
          const double2 p = tp[tid + i * nt], l = tlam[tid + i * nt];
          psi[k] = make_double2(f * p.x, f * p.y);
          lam[k] = make_double2(f * l.x, f * l.y);
        }
    }
    __syncthreads();
  }
  // one warp reduces a slot: every thread's sum in a fixed order, to the slot's op
  for (int s = tid >> 5; s < P.n_slots; s += (int)(nt >> 5)) {
    double v = 0.0;
    for (uint32_t j = tid & 31; j < nt; j += 32) v += accp[s * nt + j];
    v = warp_sum(v);
    if ((tid & 31) == 0) partial[(size_t)s_op[s] * kRedBlocks + blockIdx.x] = s_fac[s] * v;
  }
}

// Gradients only: 2 Im<lambda|G|psi> of every parameterised single-op item of the pass from
// the unchanged psi and lambda tiles (no un-apply, no stores).  Used for a commuting layer
// whose gradients are all taken at the layer's end; the tiles are read-only, so the items need
// no barrier between them.
__global__ void __launch_bounds__(kFT) k_gpass(const double2* __restrict__ psi,
                                               const double2* __restrict__ lam, FPass P,
                                               const SItem* __restrict__ items,
                                               double* __restrict__ partial) {
  extern __shared__ double2 smem[];
  __shared__ SItem its[kChunk];
  const uint32_t M = 1u << P.m, nt = blockDim.x;
  double2* tp = smem;
  double2* tlam = smem + M;
  double* accp = (double*)(smem + 2 * M);  // [n_slots][nt]
  const uint64_t ntiles = 1ull << __popcll(P.outer_mask);
  const int tid = threadIdx.x;
  const TileMap T = tile_map(P);
  items += P.first_item;
  for (int s = 0; s < P.n_slots; ++s) accp[s * nt + tid] = 0.0;
  pdl_begin();
  for (uint64_t t = blockIdx.x; t < ntiles; t += gridDim.x) {
    const uint32_t outer = pdep32((uint32_t)t, (uint32_t)P.outer_mask);
#pragma unroll
    for (int i = 0; i < 8; ++i)
      if (i < T.cnt) {
        const uint32_t k = outer | tile_idx(T, i);
        cp_async16(&tp[tid + i * nt], &psi[k]);
        cp_async16(&tlam[tid + i * nt], &lam[k]);
      }
    cp_async_wait_all();
    for (int base = 0; base < P.n_items; base += kChunk) {
      const int cnt = min(kChunk, P.n_items - base);
      if (tid < cnt) {
        its[tid] = items[base + tid];
      }
      __syncthreads();
      for (int i = 0; i < cnt; ++i) {
        const SItem& s = its[i];
        if (s.slot < 0) continue;
        const uint32_t fl = s.fl, low = fl - 1u;  // RY or RX: one bit
        double acc = 0.0;
        for (uint32_t p = tid; p < (M >> 1); p += nt) {
          const uint32_t a = ((p & ~low) << 1) | (p & low);
          const double2 px = tp[a], py = tp[a | fl], lx = tlam[a], ly = tlam[a | fl];
          if (s.kind == F_RX) fgrad<F_RX>(lx, ly, px, py, acc);
          else fgrad<F_RY>(lx, ly, px, py, acc);
        }
        accp[s.slot * nt + tid] += acc;
      }
      __syncthreads();
    }
  }
  for (int i = tid >> 5; i < P.n_items; i += (int)(nt >> 5)) {
    const int slot = items[i].slot;
    if (slot < 0) continue;
    double v = 0.0;
    for (uint32_t j = tid & 31; j < nt; j += 32) v += accp[slot * nt + j];
    v = warp_sum(v);
    if ((tid & 31) == 0) partial[(size_t)items[i].op * kRedBlocks + blockIdx.x] = v;
  }
}

}  // namespace

int fused_tile_bits() { return 11; }

namespace {
// Threads of a pass: two to eight amplitudes each, so that a small tile's gates still fill
// whole warps and no thread holds more than TileMap allows.
int pass_threads(int m) { return std::min(kFT, std::max(32, 1 << (m > 0 ? m - 1 : 0))); }
size_t fpass_smem(int m) { return ((size_t)1 << m) * sizeof(double2); }
size_t bpass_smem(int m, int slots) {
  return 2 * ((size_t)1 << m) * sizeof(double2) + (size_t)slots * pass_threads(m) * sizeof(double);
}
}  // namespace

int pass_blocks(const FPass& P) {
  const uint64_t ntiles = 1ull << __builtin_popcountll(P.outer_mask);
  return (int)std::min<uint64_t>(ntiles, kRedBlocks);
}

cudaError_t fused_prepare() {
  const int most = (int)std::max(kOnePerSm, bpass_smem(11, kMaxSlotsDev));
  const void* ks[] = {(const void*)k_fpass<false>, (const void*)k_fpass<true>,
                      (const void*)k_gpass, (const void*)k_bpass};
  for (const void* k : ks) {
    const cudaError_t e =
        cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, most);
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

namespace {
template <class... P, class... A>
cudaError_t launch_pass(void (*k)(P...), const FPass& F, size_t smem, cudaStream_t s, bool overlap,
                        A... args) {
  const int g = pass_blocks(F);
  return launch_overlapped(k, g, pass_threads(F.m), spread_smem(smem, g), s, overlap, args...);
}
}  // namespace

cudaError_t launch_fpass(double2* psi, const FPass& P, const SItem* items, const DOp* gops,
                         const double2* cs, const double* scale, cudaStream_t s, bool overlap) {
  return launch_pass(k_fpass<false>, P, fpass_smem(P.m), s, overlap, psi, P, items, gops, cs,
                     scale);
}

cudaError_t launch_fpass_inv(double2* v, const FPass& P, const SItem* items, const DOp* gops,
                             const double2* cs, const double* scale, cudaStream_t s,
                             bool overlap) {
  return launch_pass(k_fpass<true>, P, fpass_smem(P.m), s, overlap, v, P, items, gops, cs, scale);
}

cudaError_t launch_gpass(const double2* psi, const double2* lam, const FPass& P,
                         const SItem* items, double* partial, cudaStream_t s, bool overlap) {
  return launch_pass(k_gpass, P, bpass_smem(P.m, P.n_slots), s, overlap, psi, lam, P, items,
                     partial);
}

cudaError_t launch_bpass(double2* psi, double2* lam, const FPass& P, const SItem* items,
                         const DOp* gops, const double2* cs, const double* scale, double* partial,
                         cudaStream_t s, bool overlap) {
  return launch_pass(k_bpass, P, bpass_smem(P.m, P.n_slots), s, overlap, psi, lam, P, items, gops,
                     cs, scale, partial);
}

}  // namespace svqe
