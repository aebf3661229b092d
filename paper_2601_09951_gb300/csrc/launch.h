// launch.h -- host-callable launchers of the single-state kernels (k_state.cu).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "svqe_types.h"

namespace svqe {

// Fixed grid for reductions: partial arrays hold at most kRedBlocks values per launch.
constexpr int kRedBlocks = 1216;  // 152 SMs x 8
constexpr int kThreads = 256;

// Launch a kernel that calls pdl_begin so that its blocks start, and run up to pdl_begin, while
// the preceding kernel of the stream drains (programmatic dependent launch).  The gap between
// two dependent kernels and the successor's set-up (staged items, index maps) are 4 to 6 us of
// every pass over a state that sits in L2.
template <class... P, class... A>
cudaError_t launch_overlapped(void (*k)(P...), int grid, int block, size_t smem, cudaStream_t s,
                              bool overlap, A... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)grid);
  cfg.blockDim = dim3((unsigned)block);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  cfg.numAttrs = overlap ? 1 : 0;
  return cudaLaunchKernelEx(&cfg, k, static_cast<P>(args)...);
}

// Shared memory that keeps a kernel to one block per SM.  An overlapped kernel's blocks are placed
// while its predecessor's still run, so a grid of at most one block per SM would double up on the
// SMs that free first and leave others idle: at 17 qubits (128 blocks, FP64-bound) that cost
// 15 % of an evaluation.
constexpr int kSms = 152;
constexpr size_t kOnePerSm = 116 * 1024;
inline size_t spread_smem(size_t smem, int grid) {
  return grid <= kSms && smem < kOnePerSm ? kOnePerSm : smem;
}

cudaError_t launch_init_basis(double2* psi, int n, uint64_t b, cudaStream_t s);
cudaError_t launch_prep_coefs(const DOp* ops, int n_ops, const double* theta, Rot* coefs,
                              cudaStream_t s);
// Launchers below that take `overlap` must not be given it for the first kernel that reads what
// launch_prep wrote.
// Everything of a planned circuit that depends on theta, one block per unit (k_prep.cu): the
// ops' lifting coefficients, the passes' items and scales, (cos, sin) of the RZ gates and the
// phase tables (kDpTab entries each) of the whole-state segments on n qubits.
constexpr int kMaxFoldItems = 128;
cudaError_t launch_prep(const PrepUnit* units, int n_units, const DOp* ops, const FItem* items,
                        const double* theta, int n, uint64_t ref, Rot* coefs, SItem* sitems,
                        double* scales, double2* cs, double2* dptab, cudaStream_t s);
// Apply (inv = false) or un-apply one op on psi; coef points at the op's Rot.
cudaError_t launch_apply_op(double2* psi, int n, const DOp& op, const Rot* coef, bool inv,
                            cudaStream_t s, bool overlap = false);
// Adjoint step for one op: if the op is parameterised, partial[b] (b < adjoint_blocks(n, op))
// receives block b's share of 2 Im<lambda|G|psi>; then psi and lambda are un-applied.
int adjoint_blocks(int n, const DOp& op);
cudaError_t launch_adjoint_op(double2* psi, double2* lam, int n, const DOp& op, const Rot* coef,
                              double* partial, cudaStream_t s, bool overlap = false);
// lambda = H psi, and partial[b] = block b's share of Re<psi|H psi>, b < hpsi_blocks(n).
int hpsi_blocks(int n);
cudaError_t launch_hpsi(const double2* psi, double2* lam, int n, const DGroup* groups,
                        int n_groups, const double2* tables, double* partial, cudaStream_t s,
                        bool overlap = false);
// The energy alone: partial[b] = block b's share, b < kRedBlocks.
cudaError_t launch_expval(const double2* psi, int n, const DGroup* groups, int n_groups,
                          const double2* tables, double* partial, cudaStream_t s);
// out[0] = sum of partial[0..count) in a fixed order.
cudaError_t launch_sum(const double* partial, int count, double* out, cudaStream_t s);
// The end of an evaluation, in one launch: grad[p] = sum over ops l with param p (in op order)
// of sum_b partial[l * kRedBlocks + b] over the op's ops[l].flags blocks, and (epart != nullptr)
// energy[0] = the sum of epart[0..n_epart).  With theta_upd set also the descent step
// theta_upd[p] -= lr * grad[p] and (traj != nullptr) traj[0] = the energy.
cudaError_t launch_finish(const DOp* ops, int n_ops, const double* partial, int n_params,
                          double* grad, const double* epart, int n_epart, double* energy,
                          double* theta_upd, double lr, double* traj, cudaStream_t s, bool overlap = false);

}  // namespace svqe

namespace svqe {

// Fused passes of the single-state path (k_fused.cu).  Tiles of fused_tile_bits() bits (all
// of the state when it is smaller).
// Whole-state diagonal + permutation segments (k_dp.cu) are used from kDpMinQubits: below,
// a layer's RZ and CNOT gates fit one fused pass or two.
constexpr int kDpMinQubits = 11;
constexpr int kDpSmallQubits = 14, kDpMinGates = 8;  // (see plan_circuit)
int fused_tile_bits();
cudaError_t fused_prepare();
// items, scale (the pass's place) and cs as launch_prep wrote them.
cudaError_t launch_fpass(double2* psi, const FPass& P, const SItem* items, const DOp* gops,
                         const double2* cs, const double* scale, cudaStream_t s, bool overlap);
// The pass's items inverted and in reverse order, on v (un-applying the pass).
cudaError_t launch_fpass_inv(double2* v, const FPass& P, const SItem* items, const DOp* gops,
                             const double2* cs, const double* scale, cudaStream_t s,
                             bool overlap);
// Blocks a pass launches: one per tile, at most kRedBlocks.
int pass_blocks(const FPass& P);
// Whole-state diagonal + permutation segment of the single-state path (k_dp.cu): a run of
// RZ/CZ gates followed by a run of CNOT/X gates, applied in one out-of-place streaming pass
// for n >= kDpMinQubits.  The permutation P of the CNOT/X run (gates in order) is
// P(k) = c0 ^ the XOR of col[b] over the set bits b of k.
constexpr int kDpMaxRz = 32;
constexpr int kDpMaxCz = 16;
struct DpArgs {
  int n;
  uint32_t c0;
  uint32_t col[31];
  uint32_t delta;            // M^-1 e_0, M the linear part of P
  int n_cz;
  uint32_t cz_mask[kDpMaxCz];
  int n_rz;                  // parameterised RZ ops: gradient targets
  int rz_op[kDpMaxRz];
  int rz_bit[kDpMaxRz];
  const double2* tab;        // the segment's phase tables
};
// CTAs of a segment's kernels on n qubits (a power of two).
int dp_blocks(int n);
cudaError_t dp_prepare(int n);  // (attributes of the kernels an n-qubit state uses)
// log2 of the amplitudes per block of a segment's kernels on n qubits
int dp_block_log(int n);
// out[P(k)] = phase(k) in[k]
cudaError_t launch_dp_fwd(const double2* in, double2* out, const DpArgs& a, cudaStream_t s,
                          bool overlap);
// out[k] = conj(phase(k)) in[P(k)]
cudaError_t launch_dp_bwd_psi(const double2* in, double2* out, const DpArgs& a, cudaStream_t s,
                              bool overlap);
// out[k] = conj(phase(k)) lam[P(k)]; RZ gradient shares from w_k = Im(conj(out[k]) psi_b[k])
// into partial[op * kRedBlocks + block], block < dp_blocks(n)
cudaError_t launch_dp_bwd_lam(const double2* lam, const double2* psi_b, double2* out,
                              const DpArgs& a, double* partial, cudaStream_t s, bool overlap);

// The product prefix (k_dp.cu): a circuit's leading one-qubit gates on the reference state make
// a product state, and the CNOT/X run after them (if any) permutes it.  a: the run's map (the
// identity without one) and the product's tables.
// out[P(k)] = prod(k)
cudaError_t launch_prod_fwd(double2* out, const DpArgs& a, cudaStream_t s, bool overlap);
// Gradients of the prefix's parameterised ops [0, n_ops) from lambda after the run:
// partial[op * kRedBlocks] = the whole of 2 Im<lambda|G|psi>.  part: prod_scratch(n) doubles.
size_t prod_scratch(int n);
cudaError_t launch_prod_grads(const double2* lam, const DpArgs& a, const DOp* ops, int n_ops,
                              const double2* cs, uint64_t ref, double* part, double* partial,
                              cudaStream_t s, bool overlap);
constexpr int kMaxQubitGates = 64;  // gates of one qubit in a product prefix

// Gradient shares only (psi and lambda unchanged) of a pass whose items are single ops:
// partial[op * kRedBlocks + b] as for launch_bpass.
cudaError_t launch_gpass(const double2* psi, const double2* lam, const FPass& P,
                         const SItem* items, double* partial, cudaStream_t s, bool overlap);
// Backward pass: partial[op * kRedBlocks + b] receives block b's gradient share of every
// parameterised op of the pass, for the pass_blocks(P) blocks launched.
cudaError_t launch_bpass(double2* psi, double2* lam, const FPass& P, const SItem* items,
                         const DOp* gops, const double2* cs, const double* scale, double* partial,
                         cudaStream_t s, bool overlap);

// One instance of a compiled batch (device record).  steps, lr and etraj_off are used when
// BatchArgs::n_steps < 0 (per-instance step counts, as the serving loop runs them).
struct BInst {
  int32_t n, n_ops, n_groups, n_params, n_segs, n_ckpt;
  int32_t steps;
  int32_t tab_n;  // the instance's group tables: tab_n double2 entries from tab_off
  uint64_t ref;
  int64_t op_off, grp_off, theta_off, seg_off, pp_off, etraj_off;
  int64_t coef_off, contrib_off;  // scratch offsets (Rot / double units)
  int64_t grad_off;               // gradient offset (double units)
  double lr;
  int64_t tab_off;
};
static_assert(sizeof(BInst) == 128, "BInst layout");

// A work item of the batched kernel: the instances of one team class (see kClassWarps), one
// per team; unused entries of inst are -1.
struct BItem {
  int32_t cls;
  int32_t inst[8];
};
static_assert(sizeof(BItem) == 36, "BItem layout");
// Team classes of the batched kernel (8 warps per CTA): warps per team and the largest
// instance each class runs, so that every thread holds at most 16 of the 2^n amplitudes.
//   class 0: one team of 8 warps, n = 12;   class 1: two teams of 4 warps, n = 11;
//   class 2: eight teams of 1 warp, n <= 9; class 3: four teams of 2 warps, n = 10.
constexpr int kNumClasses = 4;
constexpr int kClassWarps[kNumClasses] = {8, 4, 1, 2};
constexpr int kClassQubits[kNumClasses] = {12, 11, 9, 10};

struct BatchArgs {
  const BInst* inst;
  int n_inst;
  const BItem* items;      // most expensive first
  int n_items;
  const DOp* ops;
  const DGroup* groups;
  const double2* tables;
  const Seg* segs;
  const int32_t* pptr;     // per instance n_params+1 offsets into pops (absolute)
  const int32_t* pops;     // op indices (relative to the instance) using each parameter
  double* theta;           // concatenated parameters (updated in place when n_steps != 0)
  double* energy;          // [n_inst]
  double* grad;            // concatenated gradients
  Rot* coef;               // scratch, one per op
  double* contrib;         // scratch, one per op
  double2* ckpt;           // scratch, ckpt_slot amplitudes per CTA, split evenly among teams
                           // (team_ckpt_amps per instance)
  int64_t ckpt_slot;
  int64_t smem_amps;       // dynamic shared memory per CTA, in amplitudes
  int* counter;            // work-queue head, zeroed before each launch
  int n_steps;             // 0: one evaluation; > 0: that many updates; < 0: BInst::steps
  double lr;               // step when lr_inst == nullptr (n_steps > 0)
  const double* lr_inst;   // per-instance steps, or nullptr
  double* etraj;           // energies before each update ([n_steps x n_inst], or per
                           // instance at BInst::etraj_off when n_steps < 0), or nullptr
  // Optimizer of the update step: 0 gradient descent; 1 Adam with first/second moments
  // adam_m/adam_v (indexed like grad) and t0 updates already taken.
  int opt;
  double* adam_m;
  double* adam_v;
  int adam_t0;
  double beta1, beta2, eps;
};

// A team's checkpoint scratch for an instance: n_ckpt states of 2^n amplitudes, then one block
// of kDpAuxAmps amplitudes per checkpoint slot, where a diagonal + permutation segment keeps
// the tables its forward pass built (phases, permutation, RZ slots) for the sweep to reload.
constexpr int kDpAuxAmps = 176;
inline int64_t team_ckpt_amps(int n_ckpt, int n) {
  return (int64_t)n_ckpt * ((int64_t(1) << n) + kDpAuxAmps);
}

// One instance alone, in one launch of one team (k_small): the single-state path of small
// registers.  Its records (BInst, ops, segments, parameter uses and, for host callers, theta)
// travel as a launch argument when they fit kSmallBlob bytes, else from blob_dev, and live in
// shared memory with the coefficients, so a step reads nothing from global memory but the
// Hamiltonian and its checkpoints.  Byte offsets into the blob; o_theta < 0: a.theta is used.
constexpr int kSmallBlob = 3584;
struct SmallArgs {
  BatchArgs a;  // inst, ops, segs, pptr, pops, coef and contrib are set by the kernel
  int nw;       // warps
  int n, n_ops, blob_bytes;
  int ham_bytes;  // shared memory for the Hamiltonian (a multiple of 16), or 0: read from L2
  int o_ops, o_segs, o_pptr, o_pops, o_theta;
  int n_params;
  const unsigned char* blob_dev;
  double* theta_out;  // final theta, or nullptr
  double2* ref_out;   // 2^n amplitudes that receive the reference state, or nullptr
  alignas(16) unsigned char blob[kSmallBlob];
};
static_assert(sizeof(SmallArgs) <= 4096, "the argument block stays within 4 KB");
// Warps of an n-qubit instance run alone, and the shared memory of such a launch.
int small_warps(int n);
size_t small_smem(int n, int n_ops, int n_params, int blob_bytes);
constexpr size_t kSmallSmem = 200 * 1024;
cudaError_t small_prepare();
cudaError_t launch_small(const SmallArgs& a, cudaStream_t s);

// Threads per CTA of the batched kernel and its dynamic shared memory for nmax qubits.
constexpr int kBatchThreads = 256;
constexpr int64_t kBatchSmemAmps = 2 * 4096;  // psi + lambda of one 12-qubit instance
size_t batch_smem_bytes(int nmax);
cudaError_t batch_prepare(int nmax, int* grid_out);
cudaError_t launch_batch(const BatchArgs& a, int grid, size_t smem, cudaStream_t s);

}  // namespace svqe
