// k_dp.cu -- whole-state diagonal + permutation segments of the single-state path.
//
// In a hardware-efficient layer a run of RZ (and CZ) gates is directly followed by a run of
// CNOT (and X) gates.  Fused shared-memory passes need four or more passes for such a run when
// the CNOTs chain through all qubits (a ring or a ladder), each pass moving psi and lambda
// through HBM for very little arithmetic.  Here the run is one streaming pass over the state:
//   * the CNOT/X run is an affine map of the index bits over GF(2), P(k) = c0 ^ the columns of
//     k's set bits;
//   * the diagonal part is one phase per amplitude, e^{-i sum_q phi_q s_q(k)} (times -1 for
//     the CZ gates that fire);
//   * the RZ gradients 2 Im<lambda|Z_q/2|psi> = sum_k s_q(k) w_k, w_k = Im(conj(lambda_k)
//     psi_k), are the same at either end of the diagonal part (the phase cancels in w_k), so
//     they are taken from the un-phased lambda and psi.
// A circuit's leading one-qubit gates make a product state, written and differentiated with the
// same index split (k_dp<DP_MAKE>, k_prod_lam, k_prod_fin).
// Blocks of 128 NA consecutive amplitudes are handled by 128 threads, NA (1 to 8) amplitudes
// each (k = base + tid + 128 i), so P and the phase of an amplitude split into a part per
// thread, one per i and one per block: a thread keeps its own part in registers, and the block
// and i parts of 32 rounds are tabulated together.  The phases come from tables of 128 entries over
// seven bits each (k_prep.cu).  Tables of 2048 entries staged per block (80 KB read through
// 56 KB of shared memory) cost small states ten times their work and held large ones to four
// blocks per SM: the lambda sweep took 94 us at 17 qubits and 610 us at 24, now 20 and 437.
// Out of place: the gather/scatter needs a second buffer.
//
// Bound by the FP64 pipe on an HBM-resident state (8 operations per amplitude forward, 12.75 in
// the lambda sweep, against 32 and 48 bytes).  The grid is at most 1024 blocks of 128 threads:
// seven to an SM, so all are resident and no last wave runs short.
#include <algorithm>

#include "launch.h"
#include "svqe_internal.cuh"

namespace svqe {

namespace {

constexpr int kDT = 128;       // threads per CTA
constexpr int kDTLog = kDpThreadLog;
constexpr int kChunk = 32;     // rounds tabulated at a time
constexpr int kMaxRound = 11;  // round bits (31 qubits: 2^21 blocks on 2^10 CTAs)

// The block of visit index t: bit 0 of t selects pair, bit pair_hi of t selects block bit 0,
// every other bit of t is the same block bit.  A bijection on the block indices, because pair
// has bit pair_hi set.  The amplitude P(k) ^ 1, which shares P(k)'s 32-byte sector, is
// P(k ^ delta), delta = M^-1 e_0 (M the linear part of P); pair is delta's block part, so
// adjacent CTAs read (or write) the two halves of the same sectors in the same round.
__device__ __forceinline__ uint32_t dp_block(uint32_t pair, uint32_t t) {
  if (pair <= 1u) return t;
  const uint32_t ep = 1u << (31 - __clz((int)pair));
  uint32_t b = t & ~(ep | 1u);
  if (t & 1u) b ^= pair;
  if (t & ep) b ^= 1u;
  return b;
}

__device__ __forceinline__ bool dp_cz(const DpArgs& a, uint32_t k) {
  uint32_t par = 0;
  for (int c = 0; c < a.n_cz; ++c) par ^= ((k & a.cz_mask[c]) == a.cz_mask[c]);
  return par & 1u;
}

template <int NA>
struct DpShared {
  double2 q[kChunk * NA];    // phases of the rounds' blocks times those of the i bits
  uint32_t blk[kChunk];      // the rounds' blocks and their part of P (with c0)
  uint32_t pc[kChunk];
};

// What a thread keeps for the whole launch: its part of P and of the phase.
struct DpThread {
  uint32_t pt;
  double2 ph;
};

__device__ __forceinline__ DpThread dp_start(const DpArgs& a) {
  DpThread t;
  t.ph = a.tab[threadIdx.x];
  t.pt = 0;
#pragma unroll
  for (int b = 0; b < kDTLog; ++b)
    if ((threadIdx.x >> b) & 1u) t.pt ^= a.col[b];
  return t;
}

// Tabulate rounds [r0, r0 + kChunk) of this CTA (visit indices t = blockIdx.x + r gridDim.x).
template <int NA>
__device__ __forceinline__ void dp_rounds(DpShared<NA>& S, const DpArgs& a, uint32_t r0,
                                          uint32_t nblk) {
  constexpr int BL = kDTLog + (NA == 8 ? 3 : NA == 4 ? 2 : NA == 2 ? 1 : 0);
  const int tid = threadIdx.x;
  const uint32_t pair = a.delta >> BL;
  const double2* pi = a.tab + 128;
  const double2* po = a.tab + 136;
  __syncthreads();
  for (int j = tid; j < kChunk * NA; j += kDT) {
    const int r = j / NA;
    const uint32_t t = blockIdx.x + (r0 + r) * gridDim.x;
    if (t >= nblk) break;
    const uint32_t b = dp_block(pair, t);
    if (j % NA == 0) {
      uint32_t c = a.c0;
      for (int i = BL; i < a.n; ++i)
        if ((b >> (i - BL)) & 1u) c ^= a.col[i];
      S.blk[r] = b;
      S.pc[r] = c;
    }
    double2 p = po[b & 127u];
    if (a.n > BL + 7) p = cmul(p, po[128 + ((b >> 7) & 127u)]);
    if (a.n > BL + 14) p = cmul(p, po[256 + (b >> 14)]);
    S.q[j] = NA > 1 ? cmul(p, pi[j % NA]) : p;
  }
  __syncthreads();
}

// DP_FWD: out[P(k)] = phase(k) in[k].  DP_BWD: out[k] = conj(phase(k)) in[P(k)].  DP_MAKE:
// out[P(k)] = phase(k), the tables holding the factors of a product state.
enum { DP_FWD = 0, DP_BWD = 1, DP_MAKE = 2 };
template <int NA, int MODE>
__global__ void __launch_bounds__(kDT, 7) k_dp(const double2* __restrict__ in,
                                               double2* __restrict__ out, DpArgs a) {
  __shared__ DpShared<NA> S;
  constexpr int BL = kDTLog + (NA == 8 ? 3 : NA == 4 ? 2 : NA == 2 ? 1 : 0);
  const DpThread T = dp_start(a);
  dp_rounds(S, a, 0, 1u << (a.n - BL));
  pdl_begin();
  const uint32_t nblk = 1u << (a.n - BL);
  for (uint32_t r0 = 0; blockIdx.x + r0 * gridDim.x < nblk; r0 += kChunk) {
    if (r0) dp_rounds(S, a, r0, nblk);
    for (int r = 0; r < kChunk && blockIdx.x + (r0 + r) * gridDim.x < nblk; ++r) {
      const uint32_t base = (S.blk[r] << BL) | threadIdx.x, pc = S.pc[r] ^ T.pt;
      double2 v[NA];
      if (MODE != DP_MAKE) {
#pragma unroll
        for (int i = 0; i < NA; ++i) {
          uint32_t p = pc;
#pragma unroll
          for (int b = 0; b < 3; ++b)
            if ((i >> b) & 1) p ^= a.col[kDTLog + b];
          v[i] = in[MODE == DP_BWD ? p : base | (i * kDT)];
        }
      }
#pragma unroll
      for (int i = 0; i < NA; ++i) {
        uint32_t p = pc;
#pragma unroll
        for (int b = 0; b < 3; ++b)
          if ((i >> b) & 1) p ^= a.col[kDTLog + b];
        const uint32_t k = base | (i * kDT);
        const double2 ph = cmul(T.ph, S.q[r * NA + i]);
        double2 w = ph;
        if (MODE == DP_FWD) w = cmul(v[i], ph);
        if (MODE == DP_BWD) w = cmul_conj(v[i], ph);
        if (a.n_cz && dp_cz(a, k)) w = make_double2(dneg(w.x), dneg(w.y));
        out[MODE == DP_BWD ? k : p] = w;
      }
    }
  }
}

// Backward, lambda: out[k] = conj(phase(k)) lam[P(k)], and the RZ gradient shares from
// w_k = Im(conj(out[k]) psi_b[k]) with psi_b the un-phased psi (k_dp<BWD>'s output):
// partial[op * kRedBlocks + block] for every parameterised RZ op of the segment.  The number of
// CTAs is a power of two, G: CTA c takes visit indices t = c, c + G, c + 2G, ..., so the bits of
// t below log2 G are fixed per CTA (their signs apply to the CTA's total) and the bits above
// are bits of the round r (one sum each, at most MR: 5 up to 25 qubits, which saves twelve
// registers and the spills).
template <int NA, int MR>
__global__ void __launch_bounds__(kDT, 7) k_dp_lam(const double2* __restrict__ lam,
                                                   const double2* __restrict__ psi_b,
                                                   double2* __restrict__ out, DpArgs a,
                                                   double* __restrict__ partial) {
  __shared__ DpShared<NA> S;
  __shared__ double red[kDT / 32][32];
  constexpr int NL = NA == 8 ? 3 : NA == 4 ? 2 : NA == 2 ? 1 : 0;
  constexpr int BL = kDTLog + NL;
  const DpThread T = dp_start(a);
  dp_rounds(S, a, 0, 1u << (a.n - BL));
  pdl_begin();
  const uint32_t nblk = 1u << (a.n - BL);
  const int lg = 31 - __clz((int)gridDim.x);
  const int nrb = a.n - BL - lg;  // round bits
  double W = 0.0, mid[3] = {0.0, 0.0, 0.0}, hr[MR];
#pragma unroll
  for (int b = 0; b < MR; ++b) hr[b] = 0.0;
  for (uint32_t r0 = 0; blockIdx.x + r0 * gridDim.x < nblk; r0 += kChunk) {
    if (r0) dp_rounds(S, a, r0, nblk);
    for (int r = 0; r < kChunk && blockIdx.x + (r0 + r) * gridDim.x < nblk; ++r) {
      const uint32_t base = (S.blk[r] << BL) | threadIdx.x, pc = S.pc[r] ^ T.pt;
      double wb = 0.0;
      // four slots at a time: loads first, and their sums by a partial butterfly (2.75 DADD per
      // amplitude instead of 4)
#pragma unroll
      for (int i0 = 0; i0 < NA; i0 += 4) {
        constexpr int U = NA < 4 ? NA : 4;
        double2 v[U], p[U];
        double w[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
          const int i = i0 + u;
          uint32_t src = pc;
#pragma unroll
          for (int b = 0; b < 3; ++b)
            if ((i >> b) & 1) src ^= a.col[kDTLog + b];
          v[u] = lam[src];
          p[u] = psi_b[base | (i * kDT)];
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
          const int i = i0 + u;
          const uint32_t k = base | (i * kDT);
          const double2 ph = cmul(T.ph, S.q[r * NA + i]);
          double2 x = cmul_conj(v[u], ph);
          if (a.n_cz && dp_cz(a, k)) x = make_double2(dneg(x.x), dneg(x.y));
          out[k] = x;
          w[u] = fma(x.x, p[u].y, dneg(x.y) * p[u].x);
        }
        double Sq;
        if constexpr (U == 4) {
          const double s01 = w[0] + w[1], d01 = w[0] - w[1];
          const double s23 = w[2] + w[3], d23 = w[2] - w[3];
          Sq = s01 + s23;
          mid[0] += d01 + d23;
          mid[1] += s01 - s23;
          if (NA == 8) mid[2] += i0 ? dneg(Sq) : Sq;
        } else if constexpr (U == 2) {
          Sq = w[0] + w[1];
          mid[0] += w[0] - w[1];
        } else {
          Sq = w[0];
        }
        wb += Sq;
      }
      W += wb;
#pragma unroll
      for (int b = 0; b < MR; ++b)
        if (b < nrb) hr[b] += (((r0 + r) >> b) & 1u) ? dneg(wb) : wb;
    }
  }
  // CTA totals: 0 the whole sum, 1..7 signed by a thread bit, 8..10 by an i bit, 11.. by a round
  // bit
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  {
    double v[16];
    v[0] = W;
#pragma unroll
    for (int b = 0; b < kDTLog; ++b) v[1 + b] = ((tid >> b) & 1) ? dneg(W) : W;
#pragma unroll
    for (int b = 0; b < 3; ++b) v[8 + b] = mid[b];
#pragma unroll
    for (int b = 0; b < 5; ++b) v[11 + b] = hr[b];
    const double t = warp_sum16(v);
    if ((lane & 1) == 0) red[warp][lane >> 1] = t;
  }
  if constexpr (MR > 5) {
    double v[16];
#pragma unroll
    for (int b = 0; b < 16; ++b) v[b] = b + 5 < MR ? hr[b + 5 < MR ? b + 5 : 0] : 0.0;
    const double t = warp_sum16(v);
    if ((lane & 1) == 0) red[warp][16 + (lane >> 1)] = t;
  }
  __syncthreads();
  if (tid < a.n_rz) {
    const int bit = a.rz_bit[tid];
    const uint32_t pair = a.delta >> BL;
    int j;
    bool neg = false;
    if (bit < kDTLog) {
      j = 1 + bit;
    } else if (bit < BL) {
      j = 8 + bit - kDTLog;
    } else {
      // block bit jb of the block visited at t = blockIdx.x + r G is bit src of t, flipped by
      // t's bit 0 where pair has bit jb (dp_block); bits of t below lg are the CTA's, the
      // others the round's
      const int jb = bit - BL;
      int src = jb;
      if (pair > 1u) {
        const int ph = 31 - __clz((int)pair);
        if (jb == ph) src = 0;
        else if (jb == 0) src = ph;
        neg = jb != ph && (blockIdx.x & 1u) && ((pair >> jb) & 1u);
      }
      if (src < lg) {
        j = 0;
        neg ^= (blockIdx.x >> src) & 1u;
      } else {
        j = 11 + src - lg;
      }
    }
    double v = 0.0;
#pragma unroll
    for (int w = 0; w < kDT / 32; ++w) v += red[w][j];
    // (psi and lambda carry the scale that the passes before the segment left out)
    v *= a.tab[kDpStates].x;
    partial[(size_t)a.rz_op[tid] * kRedBlocks + blockIdx.x] = neg ? dneg(v) : v;
  }
}

// ------------------------------------------------------------------------------ product prefix
// Gradients of one-qubit gates on a product state psi = prod_b f_b(k_b): with
// Lambda_b[v] = sum over k with k_b = v of lambda[k] prod_{c != b} conj f_c(k_c), a gate of qubit
// b that makes f_b's derivative g_b contributes 2 Re sum_v conj(Lambda_b[v]) g_b[v].  One pass over lambda
// replaces the un-phasing and un-applying of two states: k_prod_lam contracts it with the factors
// of all bits but the slots' (A), the threads' (B) or the blocks' (D), about 11 FP64 operations
// per amplitude against 170 for a layer of 24 RY and 24 RZ gates; k_prod_fin finishes every
// qubit from those.
//   part: A[4 CTAs][16] (a warp's 8 slots), B[CTAs][128], D[blocks][4] (a block's 4 warps).
template <int NA>
__global__ void __launch_bounds__(kDT, 4) k_prod_lam(const double2* __restrict__ lam, DpArgs a,
                                                     double* __restrict__ part) {
  __shared__ double2 so[kChunk], spi[8];
  __shared__ uint32_t sblk[kChunk], spc[kChunk];
  constexpr int BL = kDTLog + (NA == 8 ? 3 : NA == 4 ? 2 : NA == 2 ? 1 : 0);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const uint32_t nblk = 1u << (a.n - BL), pair = a.delta >> BL;
  double* pA = part;
  double2* pB = reinterpret_cast<double2*>(part + (size_t)gridDim.x * 64);
  double2* pD = pB + (size_t)gridDim.x * kDT;
  const DpThread T = dp_start(a);
  if (tid < NA) spi[tid] = a.tab[128 + tid];
  double2 A[NA], B = make_double2(0.0, 0.0);
#pragma unroll
  for (int i = 0; i < NA; ++i) A[i] = make_double2(0.0, 0.0);
  pdl_begin();
  for (uint32_t r0 = 0; blockIdx.x + r0 * gridDim.x < nblk; r0 += kChunk) {
    __syncthreads();
    const uint32_t t = blockIdx.x + (r0 + tid) * gridDim.x;
    if (tid < kChunk && t < nblk) {
      const uint32_t b = dp_block(pair, t);
      uint32_t c = a.c0;
      for (int i = BL; i < a.n; ++i)
        if ((b >> (i - BL)) & 1u) c ^= a.col[i];
      sblk[tid] = b;
      spc[tid] = c;
      double2 p = a.tab[136 + (b & 127u)];
      if (a.n > BL + 7) p = cmul(p, a.tab[264 + ((b >> 7) & 127u)]);
      if (a.n > BL + 14) p = cmul(p, a.tab[392 + (b >> 14)]);
      so[tid] = p;
    }
    __syncthreads();
    for (int r = 0; r < kChunk && blockIdx.x + (r0 + r) * gridDim.x < nblk; ++r) {
      const uint32_t pc = spc[r] ^ T.pt;
      double2 v[NA];
#pragma unroll
      for (int i = 0; i < NA; ++i) {
        uint32_t p = pc;
#pragma unroll
        for (int b = 0; b < 3; ++b)
          if ((i >> b) & 1) p ^= a.col[kDTLog + b];
        v[i] = lam[p];
      }
      const double2 o = so[r], tb = cmul(T.ph, o);
      double2 d = make_double2(0.0, 0.0);
#pragma unroll
      for (int i = 0; i < NA; ++i) {
        cmac_conj(A[i], v[i], tb);
        cmac_conj(d, v[i], spi[i]);
      }
      cmac_conj(B, d, o);
      double2 e = cmul_conj(d, T.ph);
      e.x = warp_sum(e.x);
      e.y = warp_sum(e.y);
      if (lane == 0) pD[(size_t)sblk[r] * 4 + warp] = e;
    }
  }
  double v[16];
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    v[2 * i] = i < NA ? A[i < NA ? i : 0].x : 0.0;
    v[2 * i + 1] = i < NA ? A[i < NA ? i : 0].y : 0.0;
  }
  const double t = warp_sum16(v);
  if ((lane & 1) == 0) pA[((size_t)blockIdx.x * 4 + warp) * 16 + (lane >> 1)] = t;
  pB[(size_t)blockIdx.x * kDT + tid] = B;
}

constexpr int kFT = 256;

// One CTA per qubit (index bit): Lambda_b from the parts, then the qubit's gates.
__global__ void __launch_bounds__(kFT) k_prod_fin(const double* __restrict__ part, int n_cta,
                                                  DpArgs a, int bl, const DOp* __restrict__ ops,
                                                  int n_ops, const double2* __restrict__ cs,
                                                  uint64_t ref, double* __restrict__ partial) {
  __shared__ double2 sx[kFT], st[3][128];
  __shared__ double red[kFT / 32][16];
  __shared__ double2 s_lam[2], s_cs[kMaxQubitGates];
  __shared__ int s_op[kMaxQubitGates], s_type[kMaxQubitGates], s_m;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int b = blockIdx.x, n = a.n;
  const double* pA = part;
  const double2* pB = reinterpret_cast<const double2*>(part + (size_t)n_cta * 64);
  const double2* pD = pB + (size_t)n_cta * kDT;
  const double2* f = a.tab + kDpStates;
  // this qubit's gates, in order
  if (warp == 0) {
    int m = 0;
    for (int g0 = 0; g0 < n_ops; g0 += 32) {
      const bool hit = g0 + lane < n_ops && ops[g0 + lane].bit0 == b;
      const unsigned bal = __ballot_sync(0xffffffffu, hit);
      if (hit) {
        const int j = m + __popc(bal & ((1u << lane) - 1u));
        s_op[j] = g0 + lane;
        s_type[j] = ops[g0 + lane].type;
        s_cs[j] = is_param_type(ops[g0 + lane].type) ? cs[g0 + lane] : make_double2(1.0, 0.0);
      }
      m += __popc(bal);
    }
    if (lane == 0) s_m = m;
  }
  // products of the factors of bits [b0, b1) but b
  auto others = [&](int b0, int b1, uint32_t v) {
    double2 p = make_double2(1.0, 0.0);
    for (int c = b0; c < b1; ++c, v >>= 1)
      if (c != b) p = cmul(p, f[2 * c + (v & 1u)]);
    return p;
  };
  if (b >= bl)
    for (int j = tid; j < 384; j += kFT) {
      const int b0 = bl + 7 * (j >> 7), b1 = min(b0 + 7, n);
      if (b0 < b1 && (j & 127) < (1 << (b1 - b0))) st[j >> 7][j & 127] = others(b0, b1, j & 127);
    }
  pdl_begin();
  double2 acc[2] = {make_double2(0.0, 0.0), make_double2(0.0, 0.0)};
  if (b < kDTLog) {
    double2 x = make_double2(0.0, 0.0);
    for (int c = tid >> kDTLog; c < n_cta; c += kFT / kDT) {
      const double2 v = pB[(size_t)c * kDT + (tid & (kDT - 1))];
      x.x += v.x;
      x.y += v.y;
    }
    sx[tid] = x;
    __syncthreads();
    if (tid < kDT) {
      x = make_double2(sx[tid].x + sx[tid + kDT].x, sx[tid].y + sx[tid + kDT].y);
      const double2 y = cmul_conj(x, others(0, kDTLog, tid));
      if ((tid >> b) & 1) acc[1] = y; else acc[0] = y;
    }
  } else if (b < bl) {
    double v[16];
#pragma unroll
    for (int j = 0; j < 16; ++j) v[j] = 0.0;
    for (int e = tid; e < 4 * n_cta; e += kFT)
#pragma unroll
      for (int j = 0; j < 16; ++j) v[j] += pA[(size_t)e * 16 + j];
    const double t = warp_sum16(v);
    if ((lane & 1) == 0) red[warp][lane >> 1] = t;
    __syncthreads();
    if (tid < 16) {
      double u = 0.0;
      for (int w = 0; w < kFT / 32; ++w) u += red[w][tid];
      reinterpret_cast<double*>(sx)[tid] = u;
    }
    __syncthreads();
    if (tid < (1 << (bl - kDTLog))) {
      const double2 y = cmul_conj(sx[tid], others(kDTLog, bl, tid));
      if ((tid >> (b - kDTLog)) & 1) acc[1] = y; else acc[0] = y;
    }
  } else {
    __syncthreads();
    const uint32_t nblk = 1u << (n - bl), bit = 1u << (b - bl);
    for (uint32_t k = tid; k < nblk; k += kFT) {
      double2 x = pD[(size_t)k * 4];
#pragma unroll
      for (int w = 1; w < 4; ++w) {
        const double2 y = pD[(size_t)k * 4 + w];
        x.x += y.x;
        x.y += y.y;
      }
      double2 p = st[0][k & 127u];
      if (n > bl + 7) p = cmul(p, st[1][(k >> 7) & 127u]);
      if (n > bl + 14) p = cmul(p, st[2][k >> 14]);
      if (k & bit) cmac_conj(acc[1], x, p);
      else cmac_conj(acc[0], x, p);
    }
  }
  __syncthreads();
  double w[4] = {acc[0].x, acc[0].y, acc[1].x, acc[1].y};
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    w[j] = warp_sum(w[j]);
    if (lane == 0) red[warp][j] = w[j];
  }
  __syncthreads();
  if (tid < 4) {
    double u = 0.0;
    for (int q = 0; q < kFT / 32; ++q) u += red[q][tid];
    reinterpret_cast<double*>(s_lam)[tid] = u;
  }
  __syncthreads();
  // gate j: 2 Re <Lambda, (the gates after it) (-i G_j) (the gates up to it) |ref>>
  if (tid < s_m && ops[s_op[tid]].param >= 0) {
    double2 x = make_double2(1.0, 0.0), y = make_double2(0.0, 0.0);
    if ((ref >> b) & 1ull) {
      x.x = 0.0;
      y.x = 1.0;
    }
    for (int j = 0; j < s_m; ++j) {
      qubit_apply(s_type[j], s_cs[j], x, y);
      if (j != tid) continue;
      // 2 (-i G): RY (-y, x), RX (-i y, -i x), RZ (-i x, i y)
      const double2 u = x, v = y;
      if (s_type[j] == SV_GATE_RY) {
        x = make_double2(dneg(v.x), dneg(v.y));
        y = u;
      } else if (s_type[j] == SV_GATE_RX) {
        x = make_double2(v.y, dneg(v.x));
        y = make_double2(u.y, dneg(u.x));
      } else {
        x = make_double2(u.y, dneg(u.x));
        y = make_double2(dneg(v.y), v.x);
      }
    }
    double g = s_lam[0].x * x.x;
    g = fma(s_lam[0].y, x.y, g);
    g = fma(s_lam[1].x, y.x, g);
    g = fma(s_lam[1].y, y.y, g);
    partial[(size_t)s_op[tid] * kRedBlocks] = g;
  }
}

// Amplitudes per thread: as many as leave 128 blocks, up to eight (a block's set-up costs what
// four hundred amplitudes do; one amplitude per thread in 1024 blocks took 11 us at 17 qubits).
int dp_na(int n) { return n >= 17 ? 8 : n == 16 ? 4 : n == 15 ? 2 : 1; }

}  // namespace

int dp_block_log(int n) { return kDTLog + (n >= 17 ? 3 : n == 16 ? 2 : n == 15 ? 1 : 0); }
int dp_blocks(int n) { return (int)std::min<uint64_t>(1ull << (n - dp_block_log(n)), 1024); }

template <int NA>
static cudaError_t prepare_na() {
  const void* ks[] = {(const void*)k_dp<NA, DP_FWD>, (const void*)k_dp<NA, DP_BWD>,
                      (const void*)k_dp<NA, DP_MAKE>, (const void*)k_dp_lam<NA, 5>,
                      (const void*)k_prod_lam<NA>};
  for (const void* k : ks) {
    const cudaError_t e =
        cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kOnePerSm);
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

cudaError_t dp_prepare(int n) {
  if (n < kDpMinQubits || dp_blocks(n) > kSms) return cudaSuccess;
  switch (dp_na(n)) {
    case 8: return prepare_na<8>();
    case 4: return prepare_na<4>();
    case 2: return prepare_na<2>();
    default: return prepare_na<1>();
  }
}

#define DP_LAUNCH(K, ...)                                                                     \
  switch (dp_na(a.n)) {                                                                       \
    case 8: return launch_overlapped(K(8), g, kDT, spread_smem(0, g), s, overlap, __VA_ARGS__);               \
    case 4: return launch_overlapped(K(4), g, kDT, spread_smem(0, g), s, overlap, __VA_ARGS__);               \
    case 2: return launch_overlapped(K(2), g, kDT, spread_smem(0, g), s, overlap, __VA_ARGS__);               \
    default: return launch_overlapped(K(1), g, kDT, spread_smem(0, g), s, overlap, __VA_ARGS__);              \
  }
#define DP_K_FWD(NA) k_dp<NA, DP_FWD>
#define DP_K_BWD(NA) k_dp<NA, DP_BWD>
#define DP_K_MAKE(NA) k_dp<NA, DP_MAKE>
#define DP_K_LAM(NA) k_dp_lam<NA, 5>
#define DP_K_PROD(NA) k_prod_lam<NA>

cudaError_t launch_dp_fwd(const double2* in, double2* out, const DpArgs& a, cudaStream_t s,
                          bool overlap) {
  const int g = dp_blocks(a.n);
  DP_LAUNCH(DP_K_FWD, in, out, a)
}

cudaError_t launch_dp_bwd_psi(const double2* in, double2* out, const DpArgs& a, cudaStream_t s,
                              bool overlap) {
  const int g = dp_blocks(a.n);
  DP_LAUNCH(DP_K_BWD, in, out, a)
}

cudaError_t launch_dp_bwd_lam(const double2* lam, const double2* psi_b, double2* out,
                              const DpArgs& a, double* partial, cudaStream_t s, bool overlap) {
  const int g = dp_blocks(a.n);
  if (a.n - dp_block_log(a.n) - 10 > 5)  // round bits: 1024 CTAs
    return launch_overlapped(k_dp_lam<8, kMaxRound>, g, kDT, 0, s, overlap, lam, psi_b, out, a,
                             partial);
  DP_LAUNCH(DP_K_LAM, lam, psi_b, out, a, partial)
}

cudaError_t launch_prod_fwd(double2* out, const DpArgs& a, cudaStream_t s, bool overlap) {
  const int g = dp_blocks(a.n);
  DP_LAUNCH(DP_K_MAKE, (const double2*)nullptr, out, a)
}

size_t prod_scratch(int n) {
  const size_t g = (size_t)dp_blocks(n), nblk = (size_t)1 << (n - dp_block_log(n));
  return g * 64 + g * 2 * kDT + nblk * 8;
}

static cudaError_t prod_lam(const double2* lam, const DpArgs& a, double* part, cudaStream_t s,
                            bool overlap) {
  const int g = dp_blocks(a.n);
  DP_LAUNCH(DP_K_PROD, lam, a, part)
}

cudaError_t launch_prod_grads(const double2* lam, const DpArgs& a, const DOp* ops, int n_ops,
                              const double2* cs, uint64_t ref, double* part, double* partial,
                              cudaStream_t s, bool overlap) {
  const cudaError_t e = prod_lam(lam, a, part, s, overlap);
  if (e != cudaSuccess) return e;
  return launch_overlapped(k_prod_fin, a.n, kFT, 0, s, true, (const double*)part, dp_blocks(a.n), a,
                           dp_block_log(a.n), ops, n_ops, cs, ref, partial);
}

}  // namespace svqe
