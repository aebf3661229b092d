"""GPU parity of the single-state path at the edges of its rules: registers on both sides of the
one-block limit (10 qubits; records that fit the launch's arguments and records that do not) and
of the tile rule (tiles of n - 7 bits below 18 qubits), angles on both sides of the quarter turns
where the unnormalised rotations change form, RY and RX gates that share a trip or repeat a qubit,
forward passes of more items than are staged at a time, runs of more rotations than a pass takes,
and the tile tuner's effect on psi and on the reported tile size.  (Backward passes of many items:
test_gpu_pass_limits.py.)  Tolerances as in tests/parity.py."""
import os
import subprocess
import sys

import numpy as np
import pytest

import oracle
from paper_2601_09951_gb300 import svqe
from paper_2601_09951_gb300 import workloads as W
from tests.parity import PSI_TOL, assert_energy, assert_grad

pytestmark = pytest.mark.gpu

# phi = theta / 2 on and beside the multiples of pi / 4 (form changes) and pi / 2 (zero cosine)
ANGLES = [s * (k * np.pi / 2 + d) for k in range(5) for d in (-1e-9, 0.0, 1e-9) for s in (1, -1)]


def _circuit(n, rng, n_rot, n_swap):
    """n_rot RY/RX gates on few-to-all qubits (repeats included), fixed and free, with runs of
    n_swap CNOT/X gates on the lowest qubits between them, and one of every other gate."""
    cb = W.CircuitBuilder(n)
    for q in range(n):
        cb.add(W.H, (q,))
    kinds = [W.RY, W.RY, W.RX]
    for i in range(n_rot):
        g = kinds[i // 4 % 3]
        if i % 7 == 3:
            cb.add(g, (int(rng.integers(n)),), angle=float(rng.choice(ANGLES)))
        else:
            cb.add(g, (int(rng.integers(n)),), param="new")
        if i == n_rot // 2:
            for j in range(n_swap):
                a, b = (n - 1, n - 2) if n > 1 else (0, 0)
                if j % 3 == 0 or n == 1:
                    cb.add(W.X, (a,))
                else:
                    cb.add(W.CNOT, (a, b) if j % 3 == 1 else (b, a))
    if n > 1:
        cb.add(W.CZ, (0, n - 1))
        cb.add(W.SINGLE_EXC, (n - 1, 0), param="new")
    if n > 3:
        cb.add(W.DOUBLE_EXC, (0, 1, n - 2, n - 1), param="new")
    return cb.build()


@pytest.mark.parametrize("n,n_rot,n_swap", [(1, 6, 3), (2, 9, 70), (5, 12, 33), (6, 20, 40),
                                            (7, 20, 0), (7, 150, 9), (8, 20, 3), (9, 60, 2),
                                            (10, 12, 3), (10, 120, 70), (11, 30, 8), (12, 24, 35), (13, 24, 70), (14, 20, 3),
                                            (17, 10, 40), (18, 8, 0)])
def test_pass_edges(n, n_rot, n_swap):
    rng = np.random.default_rng(900 + n)
    circ = _circuit(n, rng, n_rot, n_swap)
    theta = rng.uniform(-7, 7, circ["n_params"])
    special = rng.permutation(circ["n_params"])[: circ["n_params"] // 2]
    theta[special] = rng.choice(ANGLES, size=len(special))
    ref = int(rng.integers(1 << n))
    ctx = svqe.Context(n)
    ctx.init_reference(ref)
    ctx.apply_circuit(circ, theta)
    want = oracle.state(circ, theta, ref)
    assert np.max(np.abs(ctx.get_state() - want)) <= PSI_TOL
    if n > 14:
        # every parameter costs the oracle two to four whole energies: keep the first few
        circ = dict(circ, params=np.where(np.asarray(circ["params"]) < 5, circ["params"], -1),
                    fixed=np.where(np.asarray(circ["params"]) < 5, circ["fixed"], 0.37),
                    n_params=5)
        theta = theta[:5]
    inst = {"circuit": circ, "ham": W.random_pauli_sum(rng, n, 12, 0.5, min(4, n), 1.0),
            "ref": ref, "theta": theta}
    ctx.init_reference(ref)
    H = svqe.Ham(ctx, inst["ham"])
    e, g = ctx.adjoint_grad(circ, theta, H)
    e0, g0 = oracle.energy_grad(inst)
    assert_energy(e, e0, inst["ham"], f"n={n}")
    assert_grad(g, g0, inst["ham"], f"n={n}")


@pytest.mark.parametrize("n,layers", [(3, 1), (5, 30), (8, 2), (10, 3), (11, 2)])
def test_descent_steps_match_single_evaluations(n, layers):
    """vqe_step's trajectory (inside one launch up to 10 qubits) against adjoint_grad at each of
    its own points, and the reference state left behind."""
    inst = W.tfim_instance(n, layers)
    ctx = svqe.Context(n)
    ctx.init_reference(1)
    H = svqe.Ham(ctx, inst["ham"])
    lr = 0.3 / np.abs(inst["ham"]["coeff"]).sum()
    theta, energies = ctx.vqe_step(inst["circuit"], H, inst["theta"], lr, 6)
    ref = np.zeros(1 << n, np.complex128)
    ref[1] = 1.0
    assert np.max(np.abs(ctx.get_state() - ref)) <= PSI_TOL
    th = np.array(inst["theta"])
    for e_step in energies:
        e, g = ctx.adjoint_grad(inst["circuit"], th, H)
        assert_energy(e_step, e, inst["ham"])
        th = th - lr * g
    np.testing.assert_allclose(theta, th, rtol=0, atol=1e-11)


def _bad_records_give_nan(torch, svqe_call, rec):
    wide = rec.copy()
    wide["x_mask"][0] |= np.uint64(1) << np.uint64(40)
    e, g = svqe_call(wide)
    assert np.isnan(e) and np.all(np.isnan(g))


@pytest.mark.parametrize("make", [
    lambda: W.hea_instance(10, 4, 80, 51), lambda: W.hea_instance(11, 5, 80, 52),
    lambda: W.hea_instance(12, 5, 80, 53, ring=True), lambda: W.hea_instance(13, 4, 60, 54),
    lambda: W.hea_instance(14, 4, 60, 55, ring=True),
    lambda: W.uccsd_instance(n=13, n_elec=6, n_singles=20, n_doubles=80, n_terms=200, seed=56),
    lambda: W.uccsd_instance(n=14, n_elec=7, n_singles=56, n_doubles=200, n_terms=100, seed=57)])
def test_without_device_allocation_every_route(make):
    """The call without device allocation on both sides of the one-block limit, at its qubit and
    gate limits, against adjoint_grad; a bad record still gives NaN, and the next call is right."""
    torch = pytest.importorskip("torch")
    inst = make()
    n, theta = inst["circuit"]["n"], np.asarray(inst["theta"])
    rec, table = svqe.group_records(inst["ham"], n)
    t_d = torch.as_tensor(table.view(np.float64)).cuda()
    th_d = torch.as_tensor(theta).cuda()

    def call(records):
        g_d = torch.as_tensor(records.view(np.uint8).reshape(-1)).cuda()
        e_d = torch.zeros(1, dtype=torch.float64, device="cuda")
        gr_d = torch.zeros(len(theta), dtype=torch.float64, device="cuda")
        svqe.adjoint_grad_noalloc(inst["circuit"], inst["ref"], n, g_d.data_ptr(), len(records),
                                  t_d.data_ptr(), len(table), th_d.data_ptr(), e_d.data_ptr(),
                                  gr_d.data_ptr(), torch.cuda.current_stream().cuda_stream)
        torch.cuda.synchronize()
        return float(e_d.item()), gr_d.cpu().numpy()

    ctx = svqe.Context(n)
    ctx.init_reference(inst["ref"])
    e0, g0 = ctx.adjoint_grad(inst["circuit"], theta, svqe.Ham(ctx, inst["ham"]))
    for _ in range(2):
        _bad_records_give_nan(torch, call, rec)
        e, g = call(rec)
        assert_energy(e, e0, inst["ham"])
        assert_grad(g, g0, inst["ham"])


def test_states_the_caller_can_reach_are_not_taken_for_the_reference():
    """A circuit applied right after sv_init_reference may start from a product state; one applied
    to a state set by the caller, to an earlier circuit's result, or to a state whose address the
    caller holds (and here overwrites) may not."""
    torch = pytest.importorskip("torch")
    n = 12
    rng = np.random.default_rng(77)
    inst = W.hea_instance(n, 2, 10, 78)
    circ, theta = inst["circuit"], inst["theta"]
    ctx = svqe.Context(n)
    ctx.init_reference(5)
    ctx.apply_circuit(circ, theta)
    once = oracle.state(circ, theta, 5)
    assert np.max(np.abs(ctx.get_state() - once)) <= PSI_TOL
    ctx.apply_circuit(circ, theta)  # on its own result

    def apply(psi):
        for t, w, p, f in zip(circ["types"], circ["wires"], circ["params"], circ["fixed"]):
            wires = [int(q) for q in w[:W.N_WIRES[int(t)]]]
            psi = oracle.apply_gate(psi, n, int(t), wires, float(theta[p]) if p >= 0 else f)
        return psi

    assert np.max(np.abs(ctx.get_state() - apply(once))) <= PSI_TOL
    psi = rng.normal(size=1 << n) + 1j * rng.normal(size=1 << n)
    psi /= np.linalg.norm(psi)
    want = apply(psi)
    ctx.init_reference(5)
    ctx.set_state(psi)
    ctx.apply_circuit(circ, theta)
    assert np.max(np.abs(ctx.get_state() - want)) <= PSI_TOL
    stream = torch.cuda.current_stream().cuda_stream
    own = svqe.Context(n, stream=stream)
    ptr = own.state_ptr()
    own.init_reference(5)

    class Psi:  # the context's buffer as a torch tensor
        __cuda_array_interface__ = {"shape": (1 << n,), "typestr": "<c16", "data": (ptr, False),
                                    "version": 2}

    torch.as_tensor(Psi(), device="cuda").copy_(torch.as_tensor(psi).cuda())
    torch.cuda.synchronize()
    own.apply_circuit(circ, theta)
    assert np.max(np.abs(own.get_state() - want)) <= PSI_TOL


@pytest.mark.parametrize("n,odd", [(21, 0), (21, 1), (19, 0)])
def test_layers_of_an_odd_number_of_tile_bits(n, odd):
    """RY and RX layers planned with one low bit fewer (21 qubits: two passes instead of three;
    with one gate left out and at 19 qubits the ordinary plan).  The state against the oracle,
    three gradient entries against its parameter shift."""
    rng = np.random.default_rng(2100 + n + odd)
    cb = W.CircuitBuilder(n)
    for layer, gate in enumerate((W.RX, W.RY, W.RX)):
        for q in range(n - (odd if layer else 0)):
            cb.add(gate, (q,), param="new")
        for q in range(n):
            cb.add(W.RZ, (q,), angle=float(rng.uniform(-3, 3)))
        for q in range(n - 1):
            cb.add(W.CNOT, (q, q + 1))
    circ = cb.build()
    theta = rng.uniform(-7, 7, circ["n_params"])
    ham = W.tfim_instance(n)["ham"]
    ctx = svqe.Context(n)
    ctx.init_reference(3)
    ctx.apply_circuit(circ, theta)
    psi = oracle.state(circ, theta, 3)
    assert np.max(np.abs(ctx.get_state() - psi)) <= PSI_TOL
    H = svqe.Ham(ctx, ham)
    e, g = ctx.adjoint_grad(circ, theta, H)
    assert_energy(e, oracle.expval(psi, n, ham)[0], ham)
    which = [0, n + n // 2, circ["n_params"] - 1]
    inst = {"circuit": circ, "ham": ham, "ref": 3, "theta": theta}
    want = oracle.energy_grad_subset(inst, which)[1]
    assert_grad(g[which], [want[p] for p in which], ham)


@pytest.mark.parametrize("n,n_rot", [(6, 2200), (12, 1200), (12, 2200)])
def test_long_runs_of_fixed_rotations(n, n_rot):
    """Fixed-angle rotations take no gradient slot, and at odd multiples of a quarter turn each
    leaves out a factor of 1 / sqrt 2: all in one pass, 1024 of them would overflow the gradient
    of the free gate before them and 2048 the amplitudes.  (At 6 qubits the records of 2200 gates
    exceed the one-launch path; the CNOT first keeps the product prefix out.)  n_rot roundings of
    the angles and of the amplitudes stay below 2200 * 2^-52 = 5e-13."""
    rng = np.random.default_rng(n_rot + n)
    cb = W.CircuitBuilder(n)
    cb.add(W.CNOT, (0, 1))
    cb.add(W.RY, (2,), param="new")
    for _ in range(n_rot):
        cb.add((W.RY, W.RX)[int(rng.integers(2))], (int(rng.integers(6)),),
               angle=float((2 * rng.integers(-3, 3) + 1) * np.pi / 2))
    cb.add(W.RX, (3,), param="new")
    circ = cb.build()
    theta = rng.uniform(-3, 3, 2)
    ctx = svqe.Context(n)
    ctx.init_reference(5)
    ctx.apply_circuit(circ, theta)
    assert np.max(np.abs(ctx.get_state() - oracle.state(circ, theta, 5))) <= PSI_TOL
    inst = {"circuit": circ, "ham": W.random_pauli_sum(rng, n, 12, 0.5, 4, 1.0), "ref": 5,
            "theta": theta}
    e, g = ctx.adjoint_grad(circ, theta, svqe.Ham(ctx, inst["ham"]))
    e0, g0 = oracle.energy_grad(inst)
    assert_energy(e, e0, inst["ham"])
    assert_grad(g, g0, inst["ham"])


@pytest.mark.parametrize("first", [W.RY, W.CNOT])
def test_tuner_leaves_the_reference_state(first):
    """The tile tuner runs its candidates on psi; a call that tunes without evaluating (no descent
    steps) leaves |ref>, from which a circuit with a product prefix (RY first) and one without
    (CNOT first) both start."""
    n = 12
    cb = W.CircuitBuilder(n)
    if first == W.CNOT:
        cb.add(W.CNOT, (0, 1))
    for q in range(n):
        cb.add(W.RY, (q,), param="new")
    for q in range(n - 1):
        cb.add(W.CZ, (q, q + 1))
        cb.add(W.RX, (q,), angle=0.3 + 0.01 * first + q)
    circ = cb.build()
    theta = np.random.default_rng(41).uniform(-3, 3, circ["n_params"])
    ctx = svqe.Context(n)
    ctx.set_autotune(True)
    ctx.init_reference(5)
    ctx.vqe_step(circ, svqe.Ham(ctx, W.tfim_instance(n)["ham"]), theta, 0.1, 0)
    ref = np.zeros(1 << n, np.complex128)
    ref[5] = 1.0
    assert np.max(np.abs(ctx.get_state() - ref)) <= PSI_TOL
    ctx.apply_circuit(circ, theta)
    assert np.max(np.abs(ctx.get_state() - oracle.state(circ, theta, 5))) <= PSI_TOL


def test_tile_bits_after_a_call_in_one_launch(tmp_path):
    """Up to 10 qubits a circuit whose records fit one launch has no passes: the tuner does not run
    for it, and its tile size reads 11, not that of the last circuit that had passes (here one of
    2200 gates, for which the tuner's cache file names tiles of 2^9)."""
    code = """
import sys
import numpy as np
from paper_2601_09951_gb300 import svqe, workloads as W
n = 8
big = W.CircuitBuilder(n)
for i in range(2200):
    big.add(W.RY, (i % n,), angle=0.1 * i)
small = W.tfim_instance(n, 1)
ctx = svqe.Context(n)
ctx.set_autotune(True)
H = svqe.Ham(ctx, small["ham"])
out = []
for circ, theta in ((big.build(), np.zeros(0)), (small["circuit"], small["theta"])):
    ctx.adjoint_grad(circ, theta, H)
    out.append(ctx.tile_bits())
    ctx.vqe_step(circ, H, theta, 0.1, 2)
    out.append(ctx.tile_bits())
print("bits", *out)
"""
    cache = tmp_path / "tune.txt"
    env = dict(os.environ, SVQE_TUNE_CACHE=str(cache))

    def bits():
        run = subprocess.run([sys.executable, "-c", code], env=env, capture_output=True, text=True,
                             timeout=300, cwd=os.path.dirname(os.path.dirname(__file__)))
        assert run.returncode == 0, run.stderr
        return [int(b) for b in run.stdout.split("bits")[1].split()]

    first = bits()
    assert first[0] == first[1] and first[2:] == [11, 11]
    lines = cache.read_text().split()
    assert len(lines) == 3 and lines[0] == "8"  # one structure tuned: the large circuit's
    cache.write_text(f"8 {lines[1]} 9\n")
    assert bits() == [9, 9, 11, 11]
