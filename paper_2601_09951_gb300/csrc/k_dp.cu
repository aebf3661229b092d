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
// Blocks of 128 NA consecutive amplitudes are handled by 128 threads, NA (1 to 8) amplitudes
// each (k = base + tid + 128 i), so P and the phase of an amplitude split into a part per
// thread, one per i and one per block: a thread keeps its own part in registers, and the block
// and i parts of 32 rounds are tabulated together.  The phases come from tables of 128 entries over
// seven bits each (k_prep.cu).  Tables of 2048 entries staged per block (80 KB read through
// 56 KB of shared memory) cost small states ten times their work and held large ones to four
// blocks per SM: the lambda sweep took 94 us at 17 qubits and 610 us at 24, now 20 and 470.
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

__device__ __forceinline__ double2 cmul(const double2& a, const double2& b) {
  return make_double2(fma(a.x, b.x, dneg(a.y) * b.y), fma(a.x, b.y, a.y * b.x));
}
__device__ __forceinline__ double2 cmul_conj(const double2& a, const double2& b) {
  return make_double2(fma(a.x, b.x, a.y * b.y), fma(a.y, b.x, dneg(a.x) * b.y));
}

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

// Forward (BWD false): out[P(k)] = phase(k) in[k].  Backward: out[k] = conj(phase(k)) in[P(k)].
template <int NA, bool BWD>
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
#pragma unroll
      for (int i = 0; i < NA; ++i) {
        uint32_t p = pc;
#pragma unroll
        for (int b = 0; b < 3; ++b)
          if ((i >> b) & 1) p ^= a.col[kDTLog + b];
        v[i] = in[BWD ? p : base | (i * kDT)];
      }
#pragma unroll
      for (int i = 0; i < NA; ++i) {
        uint32_t p = pc;
#pragma unroll
        for (int b = 0; b < 3; ++b)
          if ((i >> b) & 1) p ^= a.col[kDTLog + b];
        const uint32_t k = base | (i * kDT);
        const double2 ph = cmul(T.ph, S.q[r * NA + i]);
        double2 w = BWD ? cmul_conj(v[i], ph) : cmul(v[i], ph);
        if (a.n_cz && dp_cz(a, k)) w = make_double2(dneg(w.x), dneg(w.y));
        out[BWD ? k : p] = w;
      }
    }
  }
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

// Backward, lambda: out[k] = conj(phase(k)) lam[P(k)], and the RZ gradient shares from
// w_k = Im(conj(out[k]) psi_b[k]) with psi_b the un-phased psi (k_dp<BWD>'s output):
// partial[op * kRedBlocks + block] for every parameterised RZ op of the segment.  The number of
// CTAs is a power of two, G: CTA c takes visit indices t = c, c + G, c + 2G, ..., so the bits of
// t below log2 G are fixed per CTA (their signs apply to the CTA's total) and the bits above
// are bits of the round r (one sum each, at most kMaxRound).
template <int NA>
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
  double W = 0.0, mid[3] = {0.0, 0.0, 0.0}, hr[kMaxRound];
#pragma unroll
  for (int b = 0; b < kMaxRound; ++b) hr[b] = 0.0;
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
      for (int b = 0; b < kMaxRound; ++b)
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
  if (nrb > 5) {
    double v[16];
#pragma unroll
    for (int b = 0; b < 16; ++b) v[b] = b + 5 < kMaxRound ? hr[b + 5 < kMaxRound ? b + 5 : 0] : 0.0;
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
    partial[(size_t)a.rz_op[tid] * kRedBlocks + blockIdx.x] = neg ? dneg(v) : v;
  }
}

// Amplitudes per thread: as many as leave 128 blocks, up to eight (a block's set-up costs what
// four hundred amplitudes do; one amplitude per thread in 1024 blocks took 11 us at 17 qubits).
int dp_na(int n) { return n >= 17 ? 8 : n == 16 ? 4 : n == 15 ? 2 : 1; }

}  // namespace

int dp_block_log(int n) { return kDTLog + (n >= 17 ? 3 : n == 16 ? 2 : n == 15 ? 1 : 0); }
int dp_blocks(int n) { return (int)std::min<uint64_t>(1ull << (n - dp_block_log(n)), 1024); }

cudaError_t dp_prepare() {
  const void* ks[] = {(const void*)k_dp<1, false>, (const void*)k_dp<2, false>,
                      (const void*)k_dp<4, false>, (const void*)k_dp<8, false>,
                      (const void*)k_dp<1, true>,  (const void*)k_dp<2, true>,
                      (const void*)k_dp<4, true>,  (const void*)k_dp<8, true>,
                      (const void*)k_dp_lam<1>,    (const void*)k_dp_lam<2>,
                      (const void*)k_dp_lam<4>,    (const void*)k_dp_lam<8>};
  for (const void* k : ks) {
    const cudaError_t e =
        cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kOnePerSm);
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

#define DP_LAUNCH(K, ...)                                                                     \
  switch (dp_na(a.n)) {                                                                       \
    case 8: return launch_overlapped(K(8), g, kDT, spread_smem(0, g), s, overlap, __VA_ARGS__);               \
    case 4: return launch_overlapped(K(4), g, kDT, spread_smem(0, g), s, overlap, __VA_ARGS__);               \
    case 2: return launch_overlapped(K(2), g, kDT, spread_smem(0, g), s, overlap, __VA_ARGS__);               \
    default: return launch_overlapped(K(1), g, kDT, spread_smem(0, g), s, overlap, __VA_ARGS__);              \
  }
#define DP_FWD(NA) k_dp<NA, false>
#define DP_BWD(NA) k_dp<NA, true>
#define DP_LAM(NA) k_dp_lam<NA>

cudaError_t launch_dp_fwd(const double2* in, double2* out, const DpArgs& a, cudaStream_t s,
                          bool overlap) {
  const int g = dp_blocks(a.n);
  DP_LAUNCH(DP_FWD, in, out, a)
}

cudaError_t launch_dp_bwd_psi(const double2* in, double2* out, const DpArgs& a, cudaStream_t s,
                              bool overlap) {
  const int g = dp_blocks(a.n);
  DP_LAUNCH(DP_BWD, in, out, a)
}

cudaError_t launch_dp_bwd_lam(const double2* lam, const double2* psi_b, double2* out,
                              const DpArgs& a, double* partial, cudaStream_t s, bool overlap) {
  const int g = dp_blocks(a.n);
  DP_LAUNCH(DP_LAM, lam, psi_b, out, a, partial)
}

}  // namespace svqe
