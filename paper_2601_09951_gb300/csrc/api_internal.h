// api_internal.h -- library-internal entry points shared by api.cu and serve.cu.
#pragma once

#include <cuda_runtime.h>

#include <vector>

#include "../../include/svqe.h"
#include "host_compile.h"
#include "launch.h"

namespace svqe {

// Stage a lowered circuit on a context (ops, coefficient and gradient buffers, fused plan).
// Upload a lowered circuit and plan its fused passes.  may_tune: with autotuning on
// (sv_set_autotune), a circuit structure not seen before has its tile size measured first
// (the forward pass is run on the context's psi, so only callers that re-initialise psi
// afterwards pass true).
// from_ref: psi is the reference state when the circuit runs, so that its leading one-qubit gates
// may be written as a product state.
sv_status stage_circuit(sv_ctx* c, const HostCircuit& hc, bool may_tune, bool from_ref);
// psi = |ref>, forward, lambda = H psi, adjoint sweep; stream-ordered.
sv_status adjoint_core(sv_ctx* c, const HostCircuit& hc, const sv_ham* H,
                       const double* theta_dev, double* energy_dev, double* grad_dev,
                       double* theta_upd = nullptr, double lr = 0.0, double* traj = nullptr);
// n_steps of gradient descent, enqueued on the context's stream without synchronising:
// theta_in is read before the call returns; theta_out (n_params) and energy_out (n_steps)
// are written when the stream reaches them (pinned host memory for real asynchrony).
sv_status vqe_enqueue(sv_ctx* c, const HostCircuit& hc, const sv_ham* H, const double* theta_in,
                      double lr, int32_t n_steps, double* theta_out, double* energy_out);
// Registers up to this size run in one launch of one block (see api.cu).
constexpr int kSmallQubits = 10;
// A circuit packed for launch_small: the argument block (a.ckpt, a.theta, results and the
// Hamiltonian's arrays are the caller's to set), the blob when it exceeds kSmallBlob, and the
// amplitudes of checkpoint scratch it needs.  theta (host, or nullptr) goes into the blob.
// Returns false for a register or circuit that k_small does not take.
struct SmallPack {
  SmallArgs args;
  std::vector<unsigned char> blob;
  int64_t ckpt_amps;
};
bool pack_small(const HostCircuit& hc, uint64_t ref, int n_groups, int n_table,
                const double* theta, SmallPack& out);
// Whether one block is the faster way for this circuit and a Hamiltonian of n_groups X masks, of
// which n_complex have complex tables: up to kSmallQubits qubits and not too many groups.
bool small_pays(const HostCircuit& hc, int n_groups, int n_complex);
cudaStream_t ctx_stream(sv_ctx* c);
// Keep what is staged next to psi and lambda: no third state buffer, so no whole-state segments,
// and the product prefix only where its scratch lies in psi.
void ctx_two_states(sv_ctx* c, bool on);
// Device bytes a context of hc.n > kSmallQubits qubits without checkpoints holds after a
// vqe_enqueue of hc, at most.
uint64_t ctx_request_bytes(const HostCircuit& hc, int32_t n_steps, bool two_states);
// sv_adjoint_grad_dev's evaluation with every buffer in the caller's `bytes` of device memory at
// mem (256-byte aligned), nothing allocated and nothing copied from pageable host memory.
// SV_ENOMEM, with nothing enqueued, when the circuit needs more.
sv_status adjoint_fixed(const HostCircuit& hc, uint64_t ref, const DGroup* groups, int n_groups,
                        const double2* tables, const double* theta_dev, double* energy_dev,
                        double* grad_dev, unsigned char* mem, size_t bytes, cudaStream_t s);
// Copy host bytes to the device as kernel arguments (dst 16-byte aligned, its length rounded up
// to 16 bytes): stream-ordered, and src is not read after the call.
cudaError_t put_bytes(void* dst, const void* src, size_t bytes, cudaStream_t s);
// Replace the Pauli sum held by H (lowered for c's register), reusing H's device buffers when
// they are large enough, so that a pooled context takes a new request without allocating.
sv_status ham_reload(sv_ctx* c, sv_ham* H, const sv_paulisum* h);
// True once a CUDA error has made the context unusable.
bool ctx_sticky(const sv_ctx* c);

// Layout of the batched kernel for the instances of one qubit count: the team class of their
// work items (kClassWarps) and the segment widths their circuits are cut with (segment_ops: a
// run of RY/RX gates on distinct qubits becomes a commuting-layer segment when it has at least
// min_layer gates, a run of RZ/CZ a diagonal segment when it has at least min_diag_rz RZ
// gates; shorter runs are applied gate by gate).
struct BLayout {
  int cls;
  int min_layer;
  int min_diag_rz;
};
// The fixed rule: the smallest team that holds the instance, widths 2 and 3.
BLayout default_layout(int n);

// Batched-kernel helpers: team class of an n-qubit instance under the fixed rule, teams per CTA
// of that class, work items, costliest first (cls_of_n: team class per qubit count, or
// nullptr for the fixed rule), and the FP64 flop count of one instance.
int batch_class(int n);
int class_teams(int n);
std::vector<BItem> batch_items(const std::vector<BInst>& bi, const int* cls_of_n = nullptr);
double batch_instance_flops(const HostCircuit& hc, const HostHam& hh,
                            const std::vector<Seg>& segs);

}  // namespace svqe
