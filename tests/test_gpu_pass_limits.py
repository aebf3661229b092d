"""GPU parity of the single-state path from 11 qubits at the limits of its plans: backward passes of
more items than are staged at a time (32), with the scale of their chunk kept and left to the
segment that follows (up to 128 items); the product prefix at 64 gates of a qubit and beyond;
passes that touch a part of each tile only (19 qubits and more); and evaluations of several
contexts in flight at once on streams of their own.  Tolerances as in tests/parity.py."""
import numpy as np
import pytest

import oracle
from paper_2601_09951_gb300 import svqe
from paper_2601_09951_gb300 import workloads as W
from tests.parity import PSI_TOL, assert_energy, assert_grad

pytestmark = pytest.mark.gpu


def _check(circ, theta, ham, ref, which=None):
    n = circ["n"]
    ctx = svqe.Context(n)
    ctx.init_reference(ref)
    ctx.apply_circuit(circ, theta)
    assert np.max(np.abs(ctx.get_state() - oracle.state(circ, theta, ref))) <= PSI_TOL
    e, g = ctx.adjoint_grad(circ, theta, svqe.Ham(ctx, ham))
    inst = {"circuit": circ, "ham": ham, "ref": ref, "theta": theta}
    if which is None:
        e0, g0 = oracle.energy_grad(inst)
    else:
        e0, part = oracle.energy_grad_subset(inst, which)
        g, g0 = g[which], [part[p] for p in which]
    assert_energy(e, e0, ham)
    assert_grad(g, g0, ham)


def _long_pass(cb, rng, count):
    """count gates on the five highest index bits: every kind that takes no gradient slot, a free
    gate of each kind now and then, one run of RZ."""
    free = [W.RY, W.RX, W.SINGLE_EXC, W.RZ]
    for i in range(count):
        a, b = (int(q) for q in rng.choice(5, size=2, replace=False))
        if i % (count // 8) == 0:
            g = free[i // (count // 8) % 4]
            cb.add(g, (a, b)[:W.N_WIRES[g]], param="new")
        elif i == count // 2 + 1:
            for q in range(3):
                cb.add(W.RZ, (q,), param="new")
        elif i % 4 == 0:
            cb.add(W.CZ, (a, b))
        elif i % 4 == 1:
            cb.add(W.H, (a,))
        else:
            cb.add((W.RY, W.RX)[i % 2], (a,), angle=float(rng.uniform(-7, 7)))


@pytest.mark.parametrize("n", [11, 13, 17])
@pytest.mark.parametrize("count,segment", [(33, False), (70, False), (64, True), (120, True),
                                           (150, True)])
def test_passes_of_several_staged_chunks(n, count, segment):
    rng = np.random.default_rng(1000 * n + count)
    cb = W.CircuitBuilder(n)
    cb.add(W.CNOT, (0, 1))  # (no product prefix)
    _long_pass(cb, rng, count)
    n_pass, pog = svqe.circuit_plan(cb.build())
    assert n_pass == 1 and len(pog) > 32
    if segment:
        for q in range(n):
            cb.add(W.RZ, (q,), **({"param": "new"} if q % 5 == 0 else {"angle": 0.3 + q}))
        for q in range(n - 1):
            cb.add(W.CNOT, (q, q + 1))
        cb.add(W.RY, (n - 1,), param="new")
        cb.add(W.RX, (0,), param="new")
    circ = cb.build()
    theta = rng.uniform(-7, 7, circ["n_params"])
    ham = W.random_pauli_sum(rng, n, 12, 0.5, 4, 1.0)
    _check(circ, theta, ham, int(rng.integers(1 << n)))


@pytest.mark.parametrize("n,per", [(11, 64), (11, 65), (14, 64), (15, 65)])
def test_prefix_at_the_gates_of_a_qubit_it_takes(n, per):
    rng = np.random.default_rng(n * per)
    cb = W.CircuitBuilder(n)
    kinds = [W.RY, W.H, W.RX, W.RZ, W.X]
    for i in range(per):
        for q in (0, n - 1, 3)[:3 if i % 8 == 0 else 2]:
            g = kinds[(i + q) % 5]
            if g in (W.H, W.X):
                cb.add(g, (q,))
            elif i % 16 == 1:
                cb.add(g, (q,), param="new")
            else:
                cb.add(g, (q,), angle=float(rng.uniform(-7, 7)))
    for q in range(n):
        cb.add(W.CNOT, (q, (q + 1) % n))
    cb.add(W.RY, (2,), param="new")
    circ = cb.build()
    theta = rng.uniform(-7, 7, circ["n_params"])
    _check(circ, theta, W.random_pauli_sum(rng, n, 12, 0.5, 4, 1.0), int(rng.integers(1 << n)))


@pytest.mark.parametrize("n", [18, 19, 22])
def test_passes_that_touch_a_part_of_each_tile(n):
    """Passes of CZ (one amplitude, no partner), of single CNOTs (no segment takes them) and of both
    excitations, on low, middle and high wires; at 18 qubits the whole tile is copied."""
    rng = np.random.default_rng(n)
    cb = W.CircuitBuilder(n)
    for q in range(n):
        cb.add(W.RY, (q,), param="new")
    for a, b in ((0, n - 1), (n - 2, n - 1), (3, 4), (4, 0), (1, n - 3)):
        cb.add(W.CZ, (a, b))
    cb.add(W.SINGLE_EXC, (n - 1, 2), param="new")
    for a, b in ((5, 6), (n - 1, 7), (7, n - 2), (8, 9), (2, n - 4)):
        cb.add(W.CNOT, (a, b))
        cb.add(W.CZ, (b, (b + 3) % n))
    cb.add(W.DOUBLE_EXC, (0, 1, n - 2, n - 1), param="new")
    cb.add(W.CNOT, (n - 1, 0))
    cb.add(W.SINGLE_EXC, (6, 5), param="new")
    circ = cb.build()
    theta = rng.uniform(-7, 7, circ["n_params"])
    _check(circ, theta, W.tfim_instance(n)["ham"], 3 << (n // 2), [0, n - 1, n, n + 1, n + 2])


def test_contexts_on_streams_of_their_own():
    """Evaluations of several contexts in flight at once, each on its own stream, sharing a
    Hamiltonian where the sizes agree: every result bit for bit that of the context alone."""
    torch = pytest.importorskip("torch")
    insts = [W.hea_instance(n, 3, 40, 70 + n, ring=True) for n in (8, 12, 12, 13, 16, 17)]
    work = []
    for inst in insts:
        s = torch.cuda.Stream()
        ctx = svqe.Context(inst["circuit"]["n"], stream=s.cuda_stream)
        ctx.init_reference(inst["ref"])
        th = torch.tensor(np.asarray(inst["theta"]), device="cuda")
        out = torch.zeros((21, len(th) + 1), dtype=torch.float64, device="cuda")
        work.append((ctx, svqe.Circuit(inst["circuit"]), th, svqe.Ham(ctx, inst["ham"]), out))
    work[2] = work[2][:3] + (work[1][3],) + work[2][4:]
    torch.cuda.synchronize()

    def run(w, row):
        ctx, circ, th, ham, out = w
        ctx.adjoint_grad_dev(circ, th.data_ptr(), ham, out[row].data_ptr(), out[row, 1:].data_ptr())

    for w in work:
        run(w, 0)
        torch.cuda.synchronize()
    for row in range(1, 21):
        for w in work:
            run(w, row)
    torch.cuda.synchronize()
    for w, inst in zip(work, insts):
        out = w[4].cpu().numpy()
        assert np.all(out == out[0])
        if w is not work[2]:
            e, g = oracle.energy_grad_subset(inst, [0, 1])
            assert_energy(out[0, 0], e, inst["ham"])
            assert_grad(out[0, 1:3], [g[0], g[1]], inst["ham"])


@pytest.mark.parametrize("n,terms,p_zonly", [(6, 3000, 0.2), (7, 700, 0.0), (8, 300, 0.3),
                                             (9, 260, 0.2), (9, 2000, 0.0), (10, 60, 0.5),
                                             (10, 300, 0.5), (10, 3000, 0.0)])
@pytest.mark.parametrize("layers", [1, 4])
def test_hamiltonians_on_both_sides_of_the_one_block_limit(n, terms, p_zonly, layers):
    """Up to 10 qubits a circuit runs in one block unless the Hamiltonian's groups take one SM
    longer than the passes' launches: energy, gradient, a descent step and the call without device
    allocation on either side, against the oracle and one another."""
    torch = pytest.importorskip("torch")
    rng = np.random.default_rng(n * terms + layers)
    inst = W.hea_instance(n, layers, 4, 80 + n)
    circ, theta = inst["circuit"], np.asarray(inst["theta"])
    ham = W.random_pauli_sum(rng, n, terms, p_zonly, n, 1.0)
    ctx = svqe.Context(n)
    ctx.init_reference(inst["ref"])
    H = svqe.Ham(ctx, ham)
    e, g = ctx.adjoint_grad(circ, theta, H)
    which = [0, len(theta) // 2, len(theta) - 1]
    e0, part = oracle.energy_grad_subset(dict(inst, ham=ham), which)
    assert_energy(e, e0, ham)
    assert_grad(g[which], [part[p] for p in which], ham)
    th, es = ctx.vqe_step(circ, H, theta, 0.01, 2)
    assert_energy(es[0], e, ham)
    assert_energy(es[1], ctx.adjoint_grad(circ, theta - 0.01 * g, H)[0], ham)
    rec, table = svqe.group_records(ham, n)
    bufs = [torch.as_tensor(a).cuda() for a in (rec.view(np.uint8).reshape(-1),
                                                table.view(np.float64), theta)]
    out = torch.zeros(len(theta) + 1, dtype=torch.float64, device="cuda")
    svqe.adjoint_grad_noalloc(circ, inst["ref"], n, bufs[0].data_ptr(), len(rec),
                              bufs[1].data_ptr(), len(table), bufs[2].data_ptr(), out.data_ptr(),
                              out[1:].data_ptr(), torch.cuda.current_stream().cuda_stream)
    out = out.cpu().numpy()
    assert_energy(out[0], e, ham)
    assert_grad(out[1:], g, ham)


def test_checkpointed_layer_with_a_pass_of_one_gate():
    """A layer of ten gates above the two low bits that every tile holds: passes of nine gates and
    of one, which runs as the gate's own kernel forward and as a pass in the sweep."""
    n = 19
    rng = np.random.default_rng(19)
    cb = W.CircuitBuilder(n)
    cb.add(W.CNOT, (0, n - 1))
    for gate in (W.RY, W.RX):
        for q in range(10):
            cb.add(gate, (q,), param="new")
        cb.add(W.CZ, (0, 5))
    circ = cb.build()
    n_pass, pog = svqe.circuit_plan({**circ, "types": circ["types"][1:11],
                                     "wires": circ["wires"][1:11], "params": circ["params"][1:11],
                                     "fixed": circ["fixed"][1:11]})
    assert sorted(np.bincount(pog)) == [1, 9]
    theta = rng.uniform(-7, 7, circ["n_params"])
    ham = W.tfim_instance(n)["ham"]
    inst = {"circuit": circ, "ham": ham, "ref": 77, "theta": theta}
    which = [0, 8, 9, 10, 19]
    e0, part = oracle.energy_grad_subset(inst, which)
    for budget in (0, 2 * (16 << n)):
        ctx = svqe.Context(n)
        ctx.set_checkpoint_bytes(budget)
        ctx.init_reference(77)
        e, g = ctx.adjoint_grad(circ, theta, svqe.Ham(ctx, ham))
        assert_energy(e, e0, ham)
        assert_grad(g[which], [part[p] for p in which], ham)


@pytest.mark.parametrize("n", [11, 13, 14])
@pytest.mark.parametrize("n_diag,n_perm", [(0, 2), (5, 2), (6, 2), (0, 7), (0, 8), (6, 1)])
def test_segments_of_the_fewest_gates(n, n_diag, n_perm):
    """RZ/CZ and CNOT/X runs on both sides of the least gates a whole-state segment takes, between
    layers that end up in passes."""
    rng = np.random.default_rng(n + 10 * n_diag + n_perm)
    cb = W.CircuitBuilder(n)
    cb.add(W.CNOT, (0, 1))
    for layer in range(3):
        for q in range(0, n, 2):
            cb.add((W.RY, W.RX)[layer % 2], (q,), param="new")
        for j in range(n_diag):
            if j % 3 == 2:
                cb.add(W.CZ, (j, (j + 3) % n))
            else:
                cb.add(W.RZ, (j,), param="new")
        for j in range(n_perm):
            if j % 4 == 3:
                cb.add(W.X, (j,))
            else:
                cb.add(W.CNOT, (j, (j + 1 + layer) % n))
    cb.add(W.H, (3,))
    circ = cb.build()
    theta = rng.uniform(-7, 7, circ["n_params"])
    which = [int(p) for p in rng.choice(len(theta), 6, replace=False)]
    _check(circ, theta, W.random_pauli_sum(rng, n, 12, 0.5, 4, 1.0), 3, which)
