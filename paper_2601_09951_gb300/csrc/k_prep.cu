// k_prep.cu -- what an evaluation of a planned circuit derives from its angles, in one launch.
//
// One block per fused pass, whole-state segment or product prefix.  A pass's block turns each item into the
// record the pass kernels stage (SItem), the product of the factors its RY and RX gates leave
// out into the pass's scale, and the items' gradient factors; a segment's block writes the
// segment's phase tables.  Done here once per evaluation instead of by every block of every
// pass: each block's share was a chain of about 40 FP64 instructions by one warp (1.2 us at 64
// clocks each), 10 to 20 % of a 17-qubit pass.
#include "launch.h"
#include "svqe_internal.cuh"

namespace svqe {

namespace {

constexpr int kPT = 128;

__device__ __forceinline__ int fkind_of(int type) {
  switch (type) {
    case SV_GATE_H: return F_H;
    case SV_GATE_RY: return F_RY;
    case SV_GATE_RX: return F_RX;
    case SV_GATE_SINGLE_EXC: case SV_GATE_DOUBLE_EXC: return F_EXC;
    case SV_GATE_RZ: return F_ROTZ;
    case SV_GATE_CZ: return F_NEG;
    default: return F_SWAP;
  }
}

__device__ __forceinline__ void angle_cs(const DOp* ops, int l, const double* theta, double& c,
                                         double& s) {
  const int param = ops[l].param;
  sincos(0.5 * (param >= 0 ? theta[param] : ops[l].fixed), &s, &c);
}

// The factor an item leaves out, as an unevaluated sum (1 for items that leave none).
__device__ __forceinline__ void item_factor(const FItem& it, const DOp* ops, const double* theta,
                                            double& f, double& flo) {
  f = 1.0;
  flo = 0.0;
  if (it.kind == 0 && (it.local.type == SV_GATE_RY || it.local.type == SV_GATE_RX)) {
    double c, s;
    angle_cs(ops, it.op, theta, c, s);
    const RotT t = make_rott(c, s);
    f = t.f;
    flo = t.flo;
  }
}

// Items in chunks of 128, the last chunk first (the gradient factors are products over later
// items), one thread each.  (By one warp, 32 at a time, and with the diagonal item looked for among
// the others, a pass of 150 gates took 29 us; it takes 15.)
__device__ void prep_pass(const PrepUnit& u, const DOp* ops, const FItem* items,
                          const double* theta, Rot* coefs, SItem* sitems, double* scales,
                          double2* cs) {
  constexpr int kWarps = kPT / 32;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const bool folded = u.cl > u.cf;
  __shared__ double s_f2[kPT];  // folded: f^2 of the chunk's items (at most kPT)
  __shared__ double s_w[kWarps], s_h[kWarps], s_l[kWarps];
  if (folded) {
    double f = 1.0, flo;
    if (u.cf + tid < u.cl) item_factor(items[u.cf + tid], ops, theta, f, flo);
    s_f2[tid] = f * f;
    __syncthreads();
  }
  // (cos, sin) of the diagonal item's RZ gates, by the warp least likely to have items
  if (warp == kWarps - 1 && u.diag >= 0 && lane < items[u.first + u.diag].count) {
    const int op = items[u.first + u.diag].op + lane;
    double c, s;
    angle_cs(ops, op, theta, c, s);
    cs[op] = make_double2(c, s);
  }
  double sh = 1.0, sl = 0.0, fac = 1.0;
  for (int base = (u.count - 1) / kPT * kPT; base >= 0; base -= kPT) {
    const int nw = min(kWarps, (u.count - base + 31) / 32);  // warps with items
    const int i = base + tid;
    const bool on = i < u.count;
    SItem o;
    o.p = o.q = 0.0;
    o.mode = 0;
    double nx = 1.0;
    if (warp < nw) {
      double f = 1.0, flo = 0.0;
      if (on) {
        const FItem it = items[u.first + i];
        o.lo = (uint32_t)it.local.lo_or;
        o.fl = (uint32_t)it.local.flip;
#pragma unroll
        for (int b = 0; b < 4; ++b) o.sb[b] = it.local.sb[b];
        o.k = (int16_t)it.local.k;
        o.slot = (int16_t)it.slot;
        o.op = it.op;
        o.count = it.count;
        o.kind = (int16_t)(it.kind == 1 ? F_DIAG : fkind_of(it.local.type));
        if (o.kind == F_RY || o.kind == F_RX || o.kind == F_EXC || o.kind == F_ROTZ) {
          double c, s;
          angle_cs(ops, it.op, theta, c, s);
          if (o.kind == F_RY || o.kind == F_RX) {
            const RotT t = make_rott(c, s);
            o.p = t.t;
            o.mode = (int16_t)t.mode;
            f = t.f;
            flo = t.flo;
          }
          // (a checkpointed layer's pass of one gate runs as that gate's own kernel forward)
          if (o.kind == F_EXC || o.kind == F_ROTZ || u.count == 1) {
            const Rot r = make_rot_cs(c, s);
            coefs[it.op] = r;
            if (o.kind == F_EXC || o.kind == F_ROTZ) {
              o.p = r.a;
              o.q = r.b;
              o.mode = (int16_t)r.k;
            }
          }
        }
      }
      // product of f^2 over the lanes above, and of all factors
      double w = f * f;
#pragma unroll
      for (int d = 1; d < 32; d <<= 1) {
        const double v = __shfl_down_sync(0xffffffffu, w, d);
        if (lane + d < 32) w *= v;
      }
      nx = __shfl_down_sync(0xffffffffu, w, 1);
      if (lane == 31) nx = 1.0;
#pragma unroll
      for (int d = 16; d > 0; d >>= 1) {
        const double h = __shfl_xor_sync(0xffffffffu, f, d);
        const double l = __shfl_xor_sync(0xffffffffu, flo, d);
        dd_mul(f, flo, h, l);
      }
      if (lane == 0) {
        s_w[warp] = w;
        s_h[warp] = f;
        s_l[warp] = flo;
      }
    }
    __syncthreads();
    double after = fac;
    for (int q = nw - 1; q >= 0; --q) {
      if (q > warp) after *= s_w[q];
      fac *= s_w[q];
      dd_mul(sh, sl, s_h[q], s_l[q]);
    }
    o.f = after * nx;
    if (folded && on) {
      double g = 1.0;
      for (int j = 0; j <= u.first + i - u.cf; ++j) g *= s_f2[j];
      o.f = 1.0 / g;
    }
    if (on) sitems[u.first + i] = o;
    __syncthreads();
  }
  if (tid == 0) scales[u.idx] = folded ? 1.0 : sh + sl;
}

// A pass of one gate that runs as the gate's own kernel.
__device__ void prep_coef(const PrepUnit& u, const DOp* ops, const double* theta, Rot* coefs) {
  if (threadIdx.x > 0 || !is_param_type(ops[u.first].type)) return;
  double c, s;
  angle_cs(ops, u.first, theta, c, s);
  coefs[u.first] = make_rot_cs(c, s);
}

// Index bits [b0, b1) and their values v of entry j of a segment's tables.
__device__ __forceinline__ void tab_bits(int j, int bl, int n, int& b0, int& b1, uint32_t& v) {
  if (j < 128) {
    b0 = 0; b1 = kDpThreadLog; v = j;
  } else if (j < 136) {
    b0 = kDpThreadLog; b1 = bl; v = j - 128;
  } else {
    const int t = (j - 136) >> 7;
    b0 = bl + 7 * t; b1 = min(b0 + 7, n); v = (j - 136) & 127;
  }
}

__device__ void prep_dp(const PrepUnit& u, const DOp* ops, const FItem* items,
                        const double* theta, int n, int bl, double2* tab) {
  // the product of the factors the chunk of passes before it left out
  double scale = 1.0;
  if (u.cl > u.cf) {
    __shared__ double s_h[kPT / 32], s_l[kPT / 32];
    double f = 1.0, flo = 0.0;
    if (u.cf + (int)threadIdx.x < u.cl) item_factor(items[u.cf + threadIdx.x], ops, theta, f, flo);
#pragma unroll
    for (int d = 16; d > 0; d >>= 1) {
      const double h = __shfl_xor_sync(0xffffffffu, f, d);
      const double l = __shfl_xor_sync(0xffffffffu, flo, d);
      dd_mul(f, flo, h, l);
    }
    if ((threadIdx.x & 31) == 0) {
      s_h[threadIdx.x >> 5] = f;
      s_l[threadIdx.x >> 5] = flo;
    }
    __syncthreads();
    double h = s_h[0], l = s_l[0];
#pragma unroll
    for (int w = 1; w < kPT / 32; ++w) dd_mul(h, l, s_h[w], s_l[w]);
    scale = h + l;
  }
  // (cos, sin) of the angle sum of each index bit's RZ gates
  __shared__ double2 cs[32];
  __shared__ double2 op_cs[64];
  __shared__ int op_bit[64];
  __shared__ unsigned has;
  if (threadIdx.x == 0) has = 0u;
  for (int g = threadIdx.x; g < u.count; g += kPT) {
    int bit = -1;
    if (ops[u.first + g].type == SV_GATE_RZ) {
      double c, s;
      angle_cs(ops, u.first + g, theta, c, s);
      op_cs[g] = make_double2(c, s);
      bit = ops[u.first + g].bit0;
    }
    op_bit[g] = bit;
  }
  __syncthreads();
  if ((int)threadIdx.x < n) {
    double2 p = make_double2(1.0, 0.0);
    bool any = false;
    for (int g = 0; g < u.count; ++g) {
      if (op_bit[g] != (int)threadIdx.x) continue;
      p = any ? cmul(p, op_cs[g]) : op_cs[g];
      any = true;
    }
    cs[threadIdx.x] = p;
    if (any) atomicOr(&has, 1u << threadIdx.x);
  }
  __syncthreads();
  for (int j = threadIdx.x; j < kDpStates; j += kPT) {
    int b0, b1;
    uint32_t v;
    tab_bits(j, bl, n, b0, b1, v);
    double2 p = make_double2(j < 128 ? scale : 1.0, 0.0);
    for (int b = b0; b < b1; ++b, v >>= 1)
      if ((has >> b) & 1u) p = cmul(p, make_double2(cs[b].x, v & 1u ? cs[b].y : dneg(cs[b].y)));
    tab[(size_t)u.idx * kDpTab + j] = p;
  }
  if (threadIdx.x == 0)
    tab[(size_t)u.idx * kDpTab + kDpStates] = make_double2(1.0 / (scale * scale), 0.0);
}

// The product prefix: ops [0, count) act on single qubits of the reference state, so their
// result is a product of qubit states; the tables hold products of its factors.
__device__ void prep_prod(const PrepUnit& u, const DOp* ops, const double* theta, int n, int bl,
                          uint64_t ref, double2* cs, double2* tab) {
  __shared__ double2 s_cs[kPT];
  __shared__ int s_type[kPT], s_bit[kPT];
  __shared__ double2 s_f[32][2];
  __shared__ uint8_t s_list[32][kMaxQubitGates];
  const int tid = threadIdx.x;
  double2 x = make_double2(1.0, 0.0), y = make_double2(0.0, 0.0);
  if ((ref >> (tid & 31)) & 1ull) {
    x.x = 0.0;
    y.x = 1.0;
  }
  for (int g0 = 0; g0 < u.count; g0 += kPT) {
    const int g = g0 + tid;
    __syncthreads();
    if (g < u.count) {
      double2 v = make_double2(1.0, 0.0);
      if (is_param_type(ops[g].type)) {
        angle_cs(ops, g, theta, v.x, v.y);
        cs[g] = v;
      }
      s_cs[tid] = v;
      s_type[tid] = ops[g].type;
      s_bit[tid] = ops[g].bit0;
    }
    __syncthreads();
    // each qubit's gates are listed first and then applied by all qubits at once: applied as they
    // are met, every gate would be a step of its own for the whole warp
    int m = 0;
    if (tid < n)
      for (int j = 0; j < min(kPT, u.count - g0); ++j)
        if (s_bit[j] == tid) s_list[tid][m++] = (uint8_t)j;
    for (int j = 0; j < m; ++j) qubit_apply(s_type[s_list[tid][j]], s_cs[s_list[tid][j]], x, y);
  }
  double2* t = tab + (size_t)u.idx * kDpTab;
  if (tid < n) {
    s_f[tid][0] = t[kDpStates + 2 * tid] = x;
    s_f[tid][1] = t[kDpStates + 2 * tid + 1] = y;
  }
  __syncthreads();
  for (int j = tid; j < kDpStates; j += kPT) {
    int b0, b1;
    uint32_t v;
    tab_bits(j, bl, n, b0, b1, v);
    double2 p = make_double2(1.0, 0.0);
    for (int b = b0; b < b1; ++b, v >>= 1) p = cmul(p, s_f[b][v & 1u]);
    t[j] = p;
  }
}

__global__ void __launch_bounds__(kPT) k_prep(const PrepUnit* __restrict__ units,
                                              const DOp* __restrict__ ops,
                                              const FItem* __restrict__ items,
                                              const double* __restrict__ theta, int n, int bl,
                                              uint64_t ref,
                                              Rot* __restrict__ coefs, SItem* __restrict__ sitems,
                                              double* __restrict__ scales,
                                              double2* __restrict__ cs,
                                              double2* __restrict__ dptab) {
  const PrepUnit u = units[blockIdx.x];
  if (u.kind == PREP_DP) prep_dp(u, ops, items, theta, n, bl, dptab);
  else if (u.kind == PREP_PROD) prep_prod(u, ops, theta, n, bl, ref, cs, dptab);
  else if (u.kind == PREP_COEF) prep_coef(u, ops, theta, coefs);
  else prep_pass(u, ops, items, theta, coefs, sitems, scales, cs);
}

}  // namespace

static_assert(kMaxFoldItems <= kPT, "one thread per item of a folded chunk");
static_assert(kDpMaxRz + kDpMaxCz <= 64, "a segment's diagonal ops fit prep_dp's arrays");

cudaError_t launch_prep(const PrepUnit* units, int n_units, const DOp* ops, const FItem* items,
                        const double* theta, int n, uint64_t ref, Rot* coefs, SItem* sitems,
                        double* scales, double2* cs, double2* dptab, cudaStream_t s) {
  if (n_units <= 0) return cudaSuccess;
  k_prep<<<n_units, kPT, 0, s>>>(units, ops, items, theta, n, n >= kDpMinQubits ? dp_block_log(n) : n,
                                 ref, coefs, sitems, scales, cs, dptab);
  return cudaGetLastError();
}

}  // namespace svqe
