"""What is measured: energies and gradients of variational circuits through the public calls.

A case is one call (or one short sequence of calls) of a program that uses the library: a
single state's energy and gradient, an energy alone, a few optimiser steps on one state, or a
batch of small problems.  The kinds:

  grad      Context.adjoint_grad: host angles in, energy and gradient out.
  grad_dev  Context.adjoint_grad_dev: angles, energy and gradient on the device, on torch's
            current stream (what the autograd wrapper calls).
  noalloc   adjoint_grad_noalloc: as grad_dev with every buffer the caller's.
  energy    init_reference, apply_circuit, expval: an energy without its gradient.
  steps     Context.vqe_step: gradient descent on one state.
  batch     Batch.run (host buffers) or Batch.run_dev (device buffers): energy and gradient of
            every instance.
  descent   Batch.vqe_dev or Batch.adam_dev: many optimiser steps on every instance.

The ansatz of a case is "h2" (four qubits, one DoubleExcitation, 15 terms, 100 bond lengths),
"hea" (layers of RY, RZ and a CNOT ladder), "ring" (the same with the ladder closed), "rx"
(layers of H or RX, RY, RZ and CZ), "uccsd" (Givens excitations from a Hartree-Fock state) or
"tfim" ("hea" under an Ising Hamiltonian).
"""
import math

import numpy as np
import torch

from paper_2601_09951_gb300 import svqe
from paper_2601_09951_gb300 import workloads as W


# ------------------------------------------------------------------------------------ cases
def listed():
    return [
        # One bond length of the hydrogen molecule: the smallest call, all latency.
        {"name": "h2_grad", "kind": "grad", "ansatz": "h2", "n": 4, "layers": 1, "terms": 15},
        # The hydrogen surface: every bond length's whole optimisation in one call.
        {"name": "h2_surface_adam", "kind": "descent", "ansatz": "h2", "n": 4, "layers": 1,
         "terms": 15, "count": 100, "steps": 300, "opt": "adam"},
        # A short optimisation of one eight-qubit chain.
        {"name": "tfim8_steps", "kind": "steps", "ansatz": "tfim", "n": 8, "layers": 2,
         "terms": 15, "steps": 10},
        # One mid-size state in a caller's own buffers.
        {"name": "hea11_noalloc", "kind": "noalloc", "ansatz": "hea", "n": 11, "layers": 5,
         "terms": 200},
        # One mid-size state on the device (the autograd wrapper's call).
        {"name": "hea13_grad_dev", "kind": "grad_dev", "ansatz": "hea", "n": 13, "layers": 4,
         "terms": 275},
        # An odd register whose state stays on the chip.
        {"name": "ring17_grad", "kind": "grad", "ansatz": "ring", "n": 17, "layers": 10,
         "terms": 100},
        # A molecule-shaped circuit: 400 excitations, 2000 terms.
        {"name": "uccsd20_grad", "kind": "grad", "ansatz": "uccsd", "n": 20, "layers": 400,
         "terms": 2000},
        # The scaling sweep's register that no longer fits the L2.
        {"name": "ring24_grad", "kind": "grad", "ansatz": "ring", "n": 24, "layers": 10,
         "terms": 100},
        # An energy alone (a line search, a final value) on a large register.
        {"name": "ring25_energy", "kind": "energy", "ansatz": "ring", "n": 25, "layers": 4,
         "terms": 100},
        # A handful of requests, host buffers, fewer instances than the chip has processors.
        {"name": "hea_batch60", "kind": "batch", "ansatz": "hea", "n": 0, "layers": 0,
         "terms": 0, "count": 60, "host": True},
        # The serving batch: thousands of uneven instances of 4 to 12 qubits.
        {"name": "hea_batch4096", "kind": "batch", "ansatz": "hea", "n": 0, "layers": 0,
         "terms": 0, "count": 4096, "host": False},
        # Small molecules: excitation circuits in a batch.
        {"name": "uccsd_batch150", "kind": "batch", "ansatz": "uccsd", "n": 10, "layers": 40,
         "terms": 300, "count": 150, "host": False},
    ]


def draw(rng):
    """One more case of the ranges above; none costs more than ring24_grad."""
    kind = rng.choice(["grad", "grad", "grad_dev", "noalloc", "energy", "steps", "batch",
                       "batch", "descent"])
    logi = lambda a, b: int(round(math.exp(rng.uniform(math.log(a), math.log(b)))))
    if kind == "batch":
        if rng.random() < 0.6:
            return {"kind": kind, "ansatz": "hea", "n": 0, "layers": 0, "terms": 0,
                    "count": logi(1, 4096), "host": rng.random() < 0.5}
        ans = rng.choice(["uccsd", "rx", "hea"])
        n = rng.randint(6, 12)
        return {"kind": kind, "ansatz": ans, "n": n,
                "layers": logi(10, 60) if ans == "uccsd" else rng.randint(1, 8),
                "terms": logi(20, 400), "count": logi(1, 800), "host": rng.random() < 0.5}
    if kind == "descent":
        if rng.random() < 0.5:
            return {"kind": kind, "ansatz": "h2", "n": 4, "layers": 1, "terms": 15,
                    "count": 100, "steps": logi(20, 300), "opt": rng.choice(["adam", "gd"])}
        n = rng.randint(5, 12)
        return {"kind": kind, "ansatz": "tfim", "n": n, "layers": rng.randint(1, 4),
                "terms": 2 * n - 1, "count": logi(1, 150), "steps": logi(2, 20),
                "opt": rng.choice(["adam", "gd"])}
    if kind == "steps":
        n = rng.randint(4, 18)
        return {"kind": kind, "ansatz": "tfim", "n": n, "layers": rng.randint(1, 4),
                "terms": 2 * n - 1, "steps": logi(2, 20)}
    if kind == "noalloc":
        n = rng.randint(4, 14)
        return {"kind": kind, "ansatz": rng.choice(["hea", "ring", "rx"]), "n": n,
                "layers": rng.randint(1, max(1, min(6, 240 // (4 * n)))),
                "terms": logi(20, 300)}
    ans = rng.choice(["hea", "ring", "ring", "rx", "uccsd", "tfim"])
    n = rng.randint(8, 20) if ans == "uccsd" else rng.randint(4, 24)
    most = 10 if n < 22 else 4 if ans == "rx" else 8
    layers = logi(20, 400) if ans == "uccsd" else rng.randint(1, most)
    terms = 2 * n - 1 if ans == "tfim" else logi(20, 2000 if n <= 20 else 150)
    return {"kind": kind, "ansatz": ans, "n": n, "layers": layers, "terms": terms}


# ----------------------------------------------------------------------------------- inputs
def _rng(seed, *more):
    return np.random.Generator(np.random.PCG64([int(seed), *[int(m) for m in more]]))


def _strings(rng, n, count, p_zonly, max_weight, sigma):
    """`count` random Pauli strings as masks and coefficients: a share p_zonly of Z alone, the
    others with at least one X or Y, weight 1..max_weight on distinct wires."""
    wmax = min(max_weight, n)
    wires = np.argsort(rng.random((count, n)), axis=1)[:, :wmax]
    used = np.arange(wmax)[None, :] < rng.integers(1, wmax + 1, size=(count, 1))
    zonly = rng.random(count) < p_zonly
    f = rng.integers(0, 3, size=(count, wmax))          # 0 X, 1 Y, 2 Z
    f[:, 0] = np.where(f[:, 0] == 2, rng.integers(0, 2, size=count), f[:, 0])
    f[zonly] = 2
    bit = np.left_shift(np.uint64(1), (n - 1 - wires).astype(np.uint64)) * used
    x = np.where(f <= 1, bit, 0).sum(axis=1).astype(np.uint64)
    z = np.where(f >= 1, bit, 0).sum(axis=1).astype(np.uint64)
    return {"x": x, "z": z, "coeff": rng.normal(0.0, sigma, size=count)}


def _rx_circuit(n, layers):
    """Layers of a fixed H (first layer) or RX, then RY, RZ and CZ on neighbours."""
    cb = W.CircuitBuilder(n)
    for l in range(layers):
        for q in range(n):
            if l == 0:
                cb.add(W.H, (q,))
            else:
                cb.add(W.RX, (q,), param="new")
        for q in range(n):
            cb.add(W.RY, (q,), param="new")
        for q in range(n):
            cb.add(W.RZ, (q,), param="new")
        for q in range(n - 1):
            cb.add(W.CZ, (q, q + 1))
    return cb.build()


_CIRCUITS = {}


def _hea_circuit(ansatz, n, layers):
    """Gate lists of the layered ansatz (a program builds one circuit and reuses it)."""
    key = (ansatz, n, layers)
    if key not in _CIRCUITS:
        _CIRCUITS[key] = (_rx_circuit(n, layers) if ansatz == "rx" else
                          W.hea_circuit(n, layers, ring=ansatz == "ring"))
    return _CIRCUITS[key]


def _instance(case, seed, i=0):
    """Instance i of a case: a dict as in workloads.py."""
    ans, n, layers, terms = case["ansatz"], case["n"], case["layers"], case["terms"]
    rng = _rng(seed, i)
    if ans == "uccsd":
        inst = W.uccsd_instance(n=n, n_elec=n // 2, n_singles=layers // 5,
                                n_doubles=layers - layers // 5, n_terms=terms,
                                seed=seed * 10007 + i)
        return inst
    if n == 0:  # the uneven batch: 4 to 12 qubits, 2 to 8 layers, 50 to 500 terms
        n, layers, terms = W.hea_batch_spec(i)
        ham = _strings(rng, n, terms, 0.7, 4, 0.5)
    elif ans == "tfim":
        ham = W.tfim_instance(n, layers)["ham"]
        # per-instance couplings: a field sweep
        ham = dict(ham, coeff=ham["coeff"] * (1.0 + 0.2 * rng.uniform(-1.0, 1.0)))
    elif ans == "ring":
        ham = _strings(rng, n, terms, 0.0, 6, 1.0)
    else:
        ham = _strings(rng, n, terms, 0.7, 4, 0.5)
    circ = _hea_circuit(ans, n, layers)
    return {"circuit": circ, "ham": ham, "ref": 0,
            "theta": rng.uniform(-np.pi, np.pi, size=circ["n_params"])}


def _instances(case, seed):
    if case["ansatz"] == "h2":
        if case["kind"] == "descent":
            # all start at the same small angle: the Hartree-Fock state's neighbourhood
            insts = W.h2_sweep(case["count"], seed=1000 + seed)
            for s in insts:
                s["theta"] = np.full(1, 0.01)
            return insts
        inst = W.h2_sweep(100, seed=1000 + seed)[37]
        inst["theta"] = _rng(seed).uniform(-np.pi, np.pi, size=1)
        return [inst]
    return [_instance(case, seed, i) for i in range(case.get("count", 1))]


def _lr(case, insts):
    """Optimiser step: the paper's Adam step, or a stable gradient-descent step."""
    if case.get("opt") == "adam":
        return 0.01
    return 0.4 / max(float(np.abs(s["ham"]["coeff"]).sum()) for s in insts)


def _dev(a):
    return torch.as_tensor(np.ascontiguousarray(a)).cuda()


def prepare(case, seed):
    kind = case["kind"]
    insts = _instances(case, seed)
    stream = torch.cuda.current_stream().cuda_stream
    st = {"kind": kind, "case": case}
    if kind in ("batch", "descent"):
        host = case.get("host", False)
        b = svqe.Batch(insts, stream=None if host else stream)
        st["batch"] = b
        st["theta"] = b.theta_of(insts)
        if not host:
            st["theta"] = _dev(st["theta"])
            st["energy"] = torch.empty(b.n_instances, dtype=torch.float64, device="cuda")
            st["grad"] = torch.empty(max(b.n_params, 1), dtype=torch.float64, device="cuda")
        if kind == "descent":
            st["lr"] = _lr(case, insts)
            st["traj"] = torch.empty((case["steps"], b.n_instances), dtype=torch.float64,
                                     device="cuda")
        torch.cuda.synchronize()
        return st
    inst = insts[0]
    st["circuit"] = svqe.Circuit(inst["circuit"])
    st["theta"] = inst["theta"]
    st["ref"] = inst["ref"]
    P = max(st["circuit"].n_params, 1)
    if kind in ("grad_dev", "noalloc"):
        st["theta"] = _dev(inst["theta"])
        st["energy"] = torch.empty(1, dtype=torch.float64, device="cuda")
        st["grad"] = torch.empty(P, dtype=torch.float64, device="cuda")
        st["stream"] = stream
    if kind == "noalloc":
        rec, table = svqe.group_records(inst["ham"], case["n"])
        st["n_groups"], st["n_table"] = len(rec), len(table)
        st["groups"] = torch.as_tensor(rec.view(np.uint8).reshape(-1)).cuda()
        st["tables"] = _dev(table)
    else:
        ctx = svqe.Context(case["n"], stream=stream if kind == "grad_dev" else None)
        ctx.init_reference(inst["ref"])
        st["ctx"] = ctx
        st["ham"] = svqe.Ham(ctx, inst["ham"])
    if kind == "steps":
        st["lr"] = _lr(case, insts)
    torch.cuda.synchronize()
    return st


def run(st):
    kind = st["kind"]
    if kind == "grad":
        return list(st["ctx"].adjoint_grad(st["circuit"], st["theta"], st["ham"]))
    if kind == "grad_dev":
        st["ctx"].adjoint_grad_dev(st["circuit"], st["theta"].data_ptr(), st["ham"],
                                   st["energy"].data_ptr(), st["grad"].data_ptr())
        return [st["energy"], st["grad"]]
    if kind == "noalloc":
        svqe.adjoint_grad_noalloc(st["circuit"], st["ref"], st["circuit"].n,
                                  st["groups"].data_ptr(), st["n_groups"],
                                  st["tables"].data_ptr(), st["n_table"],
                                  st["theta"].data_ptr(), st["energy"].data_ptr(),
                                  st["grad"].data_ptr(), st["stream"])
        return [st["energy"], st["grad"]]
    if kind == "energy":
        st["ctx"].init_reference(st["ref"])
        st["ctx"].apply_circuit(st["circuit"], st["theta"])
        return [st["ctx"].expval(st["ham"])]
    if kind == "steps":
        return list(st["ctx"].vqe_step(st["circuit"], st["ham"], st["theta"], st["lr"],
                                       st["case"]["steps"]))
    b = st["batch"]
    if kind == "batch":
        if st["case"]["host"]:
            return list(b.run(st["theta"]))
        b.run_dev(st["theta"].data_ptr(), st["energy"].data_ptr(), st["grad"].data_ptr())
        return [st["energy"], st["grad"]]
    theta = st["theta"].clone()
    step = b.adam_dev if st["case"]["opt"] == "adam" else b.vqe_dev
    step(theta.data_ptr(), st["lr"], st["case"]["steps"], st["traj"].data_ptr())
    return [theta, st["traj"]]


# ------------------------------------------------------------------------------------- work
def _cost(inst, grad):
    """(bytes, flops) of one evaluation: the records, angles and results once, plus psi (and
    lambda) written and read once; arithmetic gate by gate on the amplitudes a gate touches
    (a rotation 6 flops per amplitude, a run of diagonal gates 6, the sweep's un-apply of psi
    and lambda and its inner product 16 and 16), 4 per amplitude and distinct flip mask."""
    c = inst["circuit"]
    N = 2.0 ** c["n"]
    types = np.asarray(c["types"])
    flops, run = 0.0, False
    for t in types.tolist():
        amps = {W.SINGLE_EXC: N / 2, W.DOUBLE_EXC: N / 8}.get(t, N)
        diag = t in (W.RZ, W.CZ)
        if t in (W.RX, W.RY, W.SINGLE_EXC, W.DOUBLE_EXC, W.H) or (diag and not run):
            flops += amps * (22 if grad else 6)
        run = diag
    masks = len(np.unique(inst["ham"]["x"]))
    flops += N * 4 * masks
    io = 32.0 * len(types) + 24.0 * len(inst["ham"]["coeff"]) + 8.0 * c["n_params"] + 8
    if grad:
        io += 8.0 * c["n_params"]
    return io, io + 32.0 * N * (2 if grad else 1), flops


def work(case):
    kind = case["kind"]
    count = case.get("count", 1)
    if case["ansatz"] == "h2":
        sample = [W.h2_sweep(2, seed=1001)[0]]
    else:
        # the uneven batch is costed from a sample of its instances
        sample = [_instance(case, 1, i) for i in range(min(count, 64))]
    evals = case.get("steps", 1)
    io = state = flops = 0.0
    for s in sample:
        a, b, f = _cost(s, kind != "energy")
        # a batch instance lives on the chip: only its records, angles and results move
        io += a if kind in ("batch", "descent") else b
        flops += f
    scale = count / len(sample)
    if kind in ("batch", "descent"):
        return {"bytes": io * scale, "flops": flops * scale * evals}
    return {"bytes": io * scale + (evals - 1) * 8.0, "flops": flops * scale * evals}


def tolerance(case):
    # Sums of 2^n products in binary64, all of them kept in binary64.  Against plain torch one
    # evaluation measures 5e-16 to 4e-15 on the listed cases; an energy whose terms cancel
    # (1665 terms on ten qubits) 1.2e-14, and half an order more is met among drawn ones.
    # Optimiser steps measure up to 2.5e-15 over 300 steps: the descents are well conditioned.
    return {"rel": 1e-13}


# ------------------------------------------------------------------------------------ exact
def _parity(v):
    for s in (16, 8, 4, 2, 1):
        v = v ^ (v >> s)
    return (v & 1).bool()


def _view(psi, n, wire):
    """(B, 2^wire, 2, rest) view: qubit `wire` is bit n-1-wire."""
    return psi.view(psi.shape[0], 1 << wire, 2, 1 << (n - 1 - wire))


def _pair(psi, n, lo, wires):
    """The two slices of amplitudes whose bits on `wires` read lo and its complement."""
    order = sorted(range(len(wires)), key=lambda i: wires[i])
    shape, last = [psi.shape[0]], -1
    for i in order:
        shape += [1 << (wires[i] - last - 1), 2]
        last = wires[i]
    shape.append(1 << (n - 1 - last))
    v = psi.view(shape)
    a = [slice(None)] * len(shape)
    b = [slice(None)] * len(shape)
    for j, i in enumerate(order):
        a[2 + 2 * j] = lo[i]
        b[2 + 2 * j] = 1 - lo[i]
    return v[tuple(a)], v[tuple(b)]


def _bc(v, like):
    """A per-instance factor (B,) against a slice (B, ...)."""
    return v.view([-1] + [1] * (like.dim() - 1))


def _gate(psi, n, t, w, ang):
    """psi <- gate psi in place (ang: per-instance angles)."""
    if t in (W.X, W.CNOT, W.CZ, W.H):
        if t == W.CNOT:
            a, b = _pair(psi, n, (1, 0), w)[0], _pair(psi, n, (1, 1), w)[0]
        elif t == W.CZ:
            _pair(psi, n, (1, 1), w)[0].neg_()
            return
        else:
            v = _view(psi, n, w[0])
            a, b = v[:, :, 0], v[:, :, 1]
        x, y = a.clone(), b.clone()
        if t == W.H:
            r = 1.0 / math.sqrt(2.0)
            a.copy_((x + y) * r)
            b.copy_((x - y) * r)
        else:
            a.copy_(y)
            b.copy_(x)
        return
    c, s = torch.cos(ang / 2), torch.sin(ang / 2)
    if t in (W.SINGLE_EXC, W.DOUBLE_EXC):
        lo = (0, 1) if t == W.SINGLE_EXC else (0, 0, 1, 1)
        a, b = _pair(psi, n, lo, w)
    else:
        v = _view(psi, n, w[0])
        a, b = v[:, :, 0], v[:, :, 1]
    c, s = _bc(c, a), _bc(s, a)
    if t == W.RZ:
        a.mul_(torch.complex(c, -s))
        b.mul_(torch.complex(c, s))
        return
    x, y = a.clone(), b.clone()
    if t == W.RX:
        a.copy_(c * x - 1j * (s * y))
        b.copy_(c * y - 1j * (s * x))
    else:
        a.copy_(c * x - s * y)
        b.copy_(s * x + c * y)


def _inner(lam, psi, n, t, w):
    """2 Im <lam|G|psi> of a gate's generator, per instance."""
    B = psi.shape[0]
    dot = lambda u, v: (u.conj() * v).reshape(B, -1).sum(1)
    if t in (W.SINGLE_EXC, W.DOUBLE_EXC):
        lo = (0, 1) if t == W.SINGLE_EXC else (0, 0, 1, 1)
        (pa, pb), (la, lb) = _pair(psi, n, lo, w), _pair(lam, n, lo, w)
    else:
        p, l = _view(psi, n, w[0]), _view(lam, n, w[0])
        pa, pb, la, lb = p[:, :, 0], p[:, :, 1], l[:, :, 0], l[:, :, 1]
    if t == W.RZ:
        return dot(la, pa).imag - dot(lb, pb).imag
    if t == W.RX:
        return dot(la, pb).imag + dot(lb, pa).imag
    return dot(lb, pa).real - dot(la, pb).real


class _Exact:
    """Plain torch evaluation of B instances that share a circuit's gates, complex128."""

    def __init__(self, insts):
        c = insts[0]["circuit"]
        self.n, self.ref = c["n"], insts[0]["ref"]
        self.gates = list(zip(np.asarray(c["types"]).tolist(),
                              np.asarray(c["wires"]).tolist(),
                              np.asarray(c["params"]).tolist(),
                              np.asarray(c["fixed"]).tolist()))
        self.B = len(insts)
        T = max(len(s["ham"]["coeff"]) for s in insts)
        pad = lambda k, dt: np.stack([np.pad(np.asarray(s["ham"][k]).astype(dt),
                                             (0, T - len(s["ham"][k]))) for s in insts])
        self.x, self.z = _dev(pad("x", np.int64)), _dev(pad("z", np.int64))
        self.c = _dev(pad("coeff", np.float64))
        ny = np.bitwise_count(pad("x", np.uint64) & pad("z", np.uint64)) % 4
        self.phase = _dev(np.array([1, 1j, -1, -1j])[ny])

    def forward(self, theta):
        psi = torch.zeros((self.B, 1 << self.n), dtype=torch.complex128, device="cuda")
        psi[:, self.ref] = 1.0
        for t, w, p, f in self.gates:
            _gate(psi, self.n, t, w[:W.N_WIRES[t]], self._angle(theta, p, f))
        return psi

    def _angle(self, theta, p, f):
        return theta[:, p] if p >= 0 else torch.full((self.B,), f, dtype=torch.float64,
                                                     device="cuda")

    def hpsi(self, psi):
        k = torch.arange(1 << self.n, device="cuda")[None, :]
        lam = torch.zeros_like(psi)
        for t in range(self.x.shape[1]):
            src = k ^ self.x[:, t:t + 1]
            # P|j> = i^{ny} (-1)^{popc(z & j)} |j ^ x>: row k reads j = k ^ x
            f = (self.c[:, t] * self.phase[:, t])[:, None]
            v = torch.gather(psi, 1, src) * f
            lam += torch.where(_parity(src & self.z[:, t:t + 1]), -v, v)
        return lam

    def energy(self, theta):
        psi = self.forward(theta)
        return (psi.conj() * self.hpsi(psi)).sum(1).real

    def grad(self, theta):
        psi = self.forward(theta)
        lam = self.hpsi(psi)
        e = (psi.conj() * lam).sum(1).real
        g = torch.zeros_like(theta)
        for t, w, p, f in reversed(self.gates):
            w = w[:W.N_WIRES[t]]
            if p >= 0:
                g[:, p] += _inner(lam, psi, self.n, t, w)
            a = -self._angle(theta, p, f)
            _gate(psi, self.n, t, w, a)
            _gate(lam, self.n, t, w, a)
        return e, g


def exact(case, seed):
    insts = _instances(case, seed)
    kind = case["kind"]
    if kind == "batch" and case["ansatz"] == "uccsd" and \
            case["count"] * (3 * case["layers"] + case["terms"]) > 65000:
        return None  # every instance has gates of its own: one long simulation each
    # instances that share a gate list are simulated together
    groups = {}
    for i, s in enumerate(insts):
        groups.setdefault((s["circuit"]["n"], id(s["circuit"])) if kind == "batch" else 0,
                          []).append(i)
    sizes = np.cumsum([0] + [s["circuit"]["n_params"] for s in insts])
    if kind in ("steps", "descent"):
        E = _Exact(insts)
        theta = _dev(np.stack([s["theta"] for s in insts]))
        lr, traj = _lr(case, insts), []
        m, v = torch.zeros_like(theta), torch.zeros_like(theta)
        for t in range(1, case["steps"] + 1):
            e, g = E.grad(theta)
            traj.append(e)
            if case.get("opt") == "adam":
                m = 0.9 * m + (1.0 - 0.9) * g
                v = 0.999 * v + (1.0 - 0.999) * g * g
                theta = theta - lr * (m / (1.0 - 0.9 ** t)) / (
                    torch.sqrt(v / (1.0 - 0.999 ** t)) + 1e-8)
            else:
                theta = theta - lr * g
        traj = torch.stack(traj)
        if kind == "steps":
            return [theta[0].cpu().numpy(), traj[:, 0].cpu().numpy()]
        return [theta.reshape(-1), traj]
    energy = np.zeros(len(insts))
    grad = np.zeros(sizes[-1])
    for idx in groups.values():
        # chunks that keep a batch of states below a gibibyte
        per = max(1, (1 << 26) >> insts[idx[0]]["circuit"]["n"])
        for c0 in range(0, len(idx), per):
            part = idx[c0:c0 + per]
            E = _Exact([insts[i] for i in part])
            theta = _dev(np.stack([insts[i]["theta"] for i in part]))
            if kind == "energy":
                return [float(E.energy(theta)[0])]
            e, g = E.grad(theta)
            e, g = e.cpu().numpy(), g.cpu().numpy()
            for j, i in enumerate(part):
                energy[i] = e[j]
                grad[sizes[i]:sizes[i + 1]] = g[j]
    if kind == "grad":
        return [float(energy[0]), grad]
    if kind == "batch" and case["host"]:
        return [energy, grad]
    return [_dev(energy), _dev(grad)]
