"""What is timed on this library, and how its results are checked.

Every case is one call (or one forward and backward) through the public entry points of
``paper_2011_02991_gb300.qng``: a natural-gradient step of one circuit or of a batch, the metric or
the whole geometric tensor alone, the descent loop, and the energy with its autograd backward. The
sizes are those of the repository's named workloads and tests, and the odd ones between them: 4 to 16
qubits on the on-chip path, 17 to 24 on the streaming path, complex64 and complex128.

``prepare`` makes a circuit, a Hamiltonian and angles from the seed and the context that a program
keeps over its iterations; ``run`` is one iteration. ``exact`` computes the same results from their
definitions in float64 / complex128 with plain torch: the derivative states d_i psi by applying the
circuit, G_ij = <d_i psi|d_j psi> - <d_i psi|psi><psi|d_j psi>, the energy and 2 Re <psi|H|d_i psi>,
and the Tikhonov-regularised solve.
"""
import math

import numpy as np
import torch

from paper_2011_02991_gb300 import qng, workloads as W

DT, LAM = 0.1, 1e-3


# ---------------------------------------------------------------------------------------------
# the cases
def listed():
    return [
        # The smallest configuration (4 qubits, P = 16): one step is a handful of launches, so this is
        # the latency of a call, as in unit-sized studies and the inner loop of small VQE problems.
        dict(name="step_tfim4_c128", call="step", n=4, layers=2, rot="YZ", ent="CZ", ham="tfim", terms=0, prec="c128"),
        # The 12-qubit benchmark configuration (P = 192, 40 random Pauli strings) at full precision.
        dict(name="step_rand12_c128", call="step", n=12, layers=8, rot="YZ", ent="CZ", ham="random", terms=40, prec="c128"),
        # The same at complex64, the precision of long optimisations.
        dict(name="step_rand12_c64", call="step", n=12, layers=8, rot="YZ", ent="CZ", ham="random", terms=40, prec="c64"),
        # Natural-gradient VQE on the 12-site TFIM chain from small angles: ten iterations on the device.
        dict(name="optimize_vqe12_c128", call="optimize", n=12, layers=6, rot="YZ", ent="CZ", ham="tfim", terms=0,
             prec="c128", iters=10, angles="small"),
        # The whole geometric tensor of an irregular circuit (every simple gate kind at random places):
        # no layers, no runs, an odd qubit count and a ragged P.
        dict(name="qgt_ragged11_c64", call="qgt", n=11, gates=150, prec="c64"),
        # Controlled and Pauli-string rotations between ordinary gates (chemistry-style ansatz).
        dict(name="step_general11_c128", call="step", n=11, params=93, general=True, prec="c128"),
        # The metric alone at the largest on-chip size (imaginary-time evolution, Fisher-information
        # studies): 16 qubits, Ry, Rx, Rz and CNOT ladders.
        dict(name="metric16_c64", call="metric", n=16, layers=2, rot="YXZ", ent="CNOT", prec="c64"),
        # A batch of instances of uneven size (6 to 14 qubits, 2 to 10 layers, 16 to 48 strings): many
        # problems or restarts at once, where throughput counts.
        dict(name="batch64_c64", call="step", instances=64, nmin=6, nmax=14, lmax=10, prec="c64"),
        # The same at full precision.
        dict(name="batch32_c128", call="step", instances=32, nmin=6, nmax=14, lmax=10, prec="c128"),
        # <E> and its gradient through torch.autograd (plain VQE / QAOA training) on the streaming path.
        dict(name="autograd20_c64", call="autograd", n=20, layers=4, rot="YZ", ent="CZ", ham="random", terms=40, prec="c64"),
        # A full-precision step beyond the on-chip sizes: TFIM chain with site-dependent fields.
        dict(name="step_tfim22_c128", call="step", n=22, layers=2, rot="YZ", ent="CZ", ham="tfim_h", terms=0, prec="c128"),
        # The largest call: the layout of the 28-qubit benchmark (Ry, Rx, Rz, CNOT ladder, 64 random
        # strings) at 24 qubits, P = 144.
        dict(name="step_rand24_c64", call="step", n=24, layers=2, rot="YXZ", ent="CNOT", ham="random", terms=64, prec="c64"),
    ]


def draw(rng):
    """One more case: the same calls, over the whole range of sizes, layouts and precisions."""
    prec = rng.choice(("c64", "c128"))
    ham = rng.choice(("tfim", "tfim_h", "random"))
    layout = dict(rot=rng.choice(("YZ", "YXZ")), ent=rng.choice(("CZ", "CNOT")), ham=ham, terms=rng.randint(4, 64),
                  angles="uniform" if ham == "random" else "small")
    kind = rng.choice(("step", "step", "optimize", "qgt", "general", "metric", "batch", "autograd", "stream", "stream"))
    if kind == "step":
        n = rng.randint(3, 14)
        per = n * len(layout["rot"])
        return dict(call="step", n=n, layers=rng.randint(1, max(1, min(10, 240 // per))), prec=prec, **layout)
    if kind == "optimize":
        n = rng.randint(3, 12)
        return dict(call="optimize", n=n, layers=rng.randint(1, 6), iters=rng.randint(2, 10), prec="c128",
                    **dict(layout, rot="YZ", angles="small"))
    if kind == "qgt":
        return dict(call="qgt", n=rng.randint(3, 11), gates=int(20 * 8 ** rng.random()), prec=prec)
    if kind == "general":
        return dict(call="step", n=rng.randint(3, 11), params=int(8 * 12 ** rng.random()), general=True, prec=prec)
    if kind == "metric":
        n = rng.randint(6, 16 if prec == "c64" else 15)
        return dict(call="metric", n=n, layers=rng.randint(1, 3 if n < 14 else 2), prec=prec, rot=layout["rot"],
                    ent=layout["ent"])
    if kind == "batch":
        return dict(call="step", instances=int(2 * (32 if prec == "c64" else 16) ** rng.random()), nmin=rng.randint(3, 6),
                    nmax=rng.randint(8, 14), lmax=rng.randint(3, 10), prec=prec)
    if kind == "autograd":
        return dict(call="autograd", n=rng.randint(17, 20), layers=rng.randint(1, 4), prec=prec, **layout)
    n = rng.randint(17, 23 if prec == "c64" else 21)
    per = n * len(layout["rot"])
    return dict(call="step", n=n, layers=rng.randint(1, max(1, min(3, 140 // per))), prec=prec, **layout)


# ---------------------------------------------------------------------------------------------
# problems
def _layered(case, rng):
    n = case["n"]
    kinds = tuple({"X": W.RX, "Y": W.RY, "Z": W.RZ}[r] for r in case["rot"])
    c = W.layered_ansatz(n, case["layers"], kinds, W.CZ if case["ent"] == "CZ" else W.CNOT)
    ham = case.get("ham")
    if ham == "tfim":
        h = W.tfim_chain(n, 1.0, 0.7)
    elif ham == "tfim_h":
        h = W.tfim_chain(n, 1.0, rng.uniform(0.2, 1.0, n))
    else:
        h = _random_hamiltonian(n, case.get("terms", 0), rng)
    return c, h


def _instance_sizes(case):
    """(n, layers, terms) of every instance of a batch: uneven, and the same whatever the seed."""
    rng = np.random.Generator(np.random.PCG64([case["instances"], case["nmin"], case["nmax"], case["lmax"]]))
    return [(int(rng.integers(case["nmin"], case["nmax"] + 1)), int(rng.integers(2, case["lmax"] + 1)),
             int(rng.integers(16, 49))) for _ in range(case["instances"])]


def _random_hamiltonian(n, terms, rng):
    """Random strings and the constant (core) energy that qubit Hamiltonians carry as an identity term."""
    h = W.random_pauli_hamiltonian(n, terms, rng)
    zero = np.zeros(1, dtype=np.uint64)
    return W.Hamiltonian(np.append(h.coeffs, -1.0 - 0.5 * math.sqrt(terms)), np.append(h.xmask, zero), np.append(h.zmask, zero))


def _irregular_circuit(case):
    """The circuit of a case without layers: drawn from the case's own number, the same for every seed."""
    if case["call"] == "qgt":
        return W.random_circuit(case["n"], case["gates"], np.random.Generator(np.random.PCG64([case["n"], case["gates"]])))
    return W.general_problem(case["n"], case["params"], 1000 * case["n"] + case["params"]).circuit


def _problems(case, seed):
    prec = W.C64 if case["prec"] == "c64" else W.C128
    rng = np.random.Generator(np.random.PCG64([20110299, int(seed)]))
    if "instances" in case:
        out = []
        for n, layers, terms in _instance_sizes(case):
            c = W.layered_ansatz(n, layers)
            h = _random_hamiltonian(n, terms, rng)
            out.append(W.Problem("instance", c, h, W.uniform_theta(c.num_params, rng), dt=DT, lam=LAM, precision=prec))
        return out
    if case["call"] == "qgt" or case.get("general"):
        c = _irregular_circuit(case)
        h = _random_hamiltonian(case["n"], 2 * case["n"], rng)
    else:
        c, h = _layered(case, rng)
    theta = W.uniform_theta(c.num_params, rng)
    if case.get("angles") == "small":  # the start of a descent, near the product state
        theta = rng.uniform(-0.2, 0.2, c.num_params)
    return [W.Problem("case", c, h, theta, dt=DT, lam=LAM, precision=prec)]


def prepare(case, seed):
    problems = _problems(case, seed)
    ctx = qng.Context(problems if len(problems) > 1 else problems[0])
    return {"case": case, "ctx": ctx, "theta": ctx.theta0()}


def run(state):
    case, ctx, theta = state["case"], state["ctx"], state["theta"]
    call = case["call"]
    if call == "step":
        o = ctx.step(theta, DT, LAM)
        return {k: o[k] for k in ("g", "grad", "energy", "dtheta")}
    if call == "metric":
        g, sigma = ctx.metric(theta, want_sigma=True)
        return {"g": g, "sigma": sigma}
    if call == "qgt":
        return {"G": ctx.metric_complex(theta)}
    if call == "optimize":
        theta = theta.clone()
        energies = ctx.optimize(theta, DT, LAM, case["iters"])
        return {"theta": theta, "energies": energies}
    theta = theta.clone().requires_grad_(True)
    e = qng.energy(theta, ctx)
    e.sum().backward()
    return {"energy": e.detach(), "grad": theta.grad}


# ---------------------------------------------------------------------------------------------
def _sizes(case):
    """(n, P, Hamiltonian terms) of every instance."""
    if "instances" in case:
        return [(n, 2 * n * layers, terms + 1) for n, layers, terms in _instance_sizes(case)]
    n = case["n"]
    if case["call"] == "qgt" or case.get("general"):
        return [(n, _irregular_circuit(case).num_params, 2 * n + 1)]
    terms = case.get("terms", 0) + 1 if case.get("ham") == "random" else 2 * n - 1
    return [(n, n * len(case["rot"]) * case["layers"], terms)]


def work(case):
    """Bytes: angles in, results out. Flops: of every metric element one real inner product over the
    state (4 per amplitude) and one adjoint rotation of the column (4), both for i < j; the forward
    sweep and the reverse sweep at 4 per rotation and amplitude (two states in the reverse sweep, with
    its inner product); 8 per Hamiltonian term and amplitude."""
    nbytes = flops = 0.0
    call = case["call"]
    for n, P, terms in _sizes(case):
        N = float(1 << n)
        times = case.get("iters", 1)
        fwd = 4 * N * P
        rev = 12 * N * P + 8 * N * terms
        met = 8 * N * P * (P - 1) / 2
        if call == "qgt":
            met += 4 * N * P * (P - 1) / 2
        if call == "autograd":
            flops += 2 * fwd + rev + 8 * N * terms
            nbytes += 8 * (3 * P + 2)
        else:
            flops += times * (fwd + met + (0 if call in ("qgt", "metric") else rev + P ** 3 / 3))
            nbytes += times * 8 * (P + {"step": P * P + 2 * P + 1, "metric": P * P + P, "qgt": 2 * P * P, "optimize": P + 1}[call])
    return {"bytes": nbytes, "flops": flops}


def tolerance(case):
    """Relative 2-norm error that rounding leaves, about four times the largest seen against ``exact``
    over 50 drawn cases. The step solves (g + lam I) dtheta = -dt grad with lam = 1e-3, which multiplies
    the errors of g and grad by up to cond(g + lam I), 1e3 and more: dtheta 6e-4 (complex64) and 1e-12
    (complex128; 1e-11 after ten iterations of the loop), g, grad and <E> 3e-6 and 5e-14."""
    if case["prec"] == "c128":
        return {"rel": 5e-11} if case["call"] in ("step", "optimize") else {"rel": 1e-13}
    return {"rel": 2.5e-3} if case["call"] == "step" else {"rel": 1.2e-5}


# ---------------------------------------------------------------------------------------------
# the same results from their definitions, complex128
def _dev():
    return torch.device("cuda" if torch.cuda.is_available() else "cpu")


def _pauli_apply(x, n, xmask, zmask):
    """sigma x for a stack x of states (k, 2^n): sigma |m> = i^ny (-1)^popcount(m & z) |m ^ x>."""
    m = torch.arange(1 << n, device=x.device)
    src = m ^ xmask
    par = torch.zeros_like(m)
    for q in range(n):
        if (zmask >> q) & 1:
            par ^= (src >> q) & 1
    ph = (1j) ** (bin(xmask & zmask).count("1") % 4)
    return x[:, src] * ((1 - 2 * par).to(x.dtype) * ph)


def _sigma(x, n, axis, q):
    """A one-qubit Pauli on qubit q of a stack of states."""
    v = x.view(x.shape[0], 1 << (n - 1 - q), 2, 1 << q)
    y = torch.empty_like(v)
    a, b = v[:, :, 0], v[:, :, 1]
    if axis == W.RX:
        y[:, :, 0], y[:, :, 1] = b, a
    elif axis == W.RY:
        y[:, :, 0], y[:, :, 1] = b * -1j, a * 1j
    else:
        y[:, :, 0], y[:, :, 1] = a, -b
    return y.view(x.shape)


def _generator(x, n, kind, q0, q1, masks):
    """K x: the operator that generates a rotation (a Pauli string, or its controlled projection)."""
    if kind in W.SIMPLE_ROTATIONS:
        return _sigma(x, n, kind, q0)
    if kind in (W.CRX, W.CRY, W.CRZ):
        y = _sigma(x, n, {W.CRX: W.RX, W.CRY: W.RY, W.CRZ: W.RZ}[kind], q1)
    else:
        y = _pauli_apply(x, n, int(masks[0]), int(masks[1]))
    if kind != W.RP:
        y = y * ((torch.arange(1 << n, device=x.device) >> q0) & 1).to(x.dtype)
    return y


def _rotate(x, n, kind, q0, q1, masks, theta):
    c, s = math.cos(theta / 2), math.sin(theta / 2)
    kx = _generator(x, n, kind, q0, q1, masks)
    if kind in W.SIMPLE_ROTATIONS or kind == W.RP:  # K^2 = 1
        x.mul_(c)
    else:  # K^2 = |1><1| on the control: identity where it is 0
        x.mul_(1 + (c - 1) * ((torch.arange(1 << n, device=x.device) >> q0) & 1).to(x.dtype))
    return x.add_(kx, alpha=-1j * s)


def _fixed(x, n, kind, q0, q1):
    if kind in (W.X, W.Y, W.Z):
        return x.copy_(_sigma(x, n, {W.X: W.RX, W.Y: W.RY, W.Z: W.RZ}[kind], q0))
    if kind == W.H:
        return x.copy_((_sigma(x, n, W.RX, q0) + _sigma(x, n, W.RZ, q0)) * math.sqrt(0.5))
    lo, hi = min(q0, q1), max(q0, q1)
    v = x.view(x.shape[0], 1 << (n - 1 - hi), 2, 1 << (hi - lo - 1), 2, 1 << lo)
    if kind == W.CZ:
        v[:, :, 1, :, 1].neg_()
    else:  # CNOT: control q0, target q1
        a, b = (v[:, :, 1, :, 0], v[:, :, 1, :, 1]) if q0 == hi else (v[:, :, 0, :, 1], v[:, :, 1, :, 1])
        t = a.clone()
        a.copy_(b)
        b.copy_(t)
    return x


def _stack(circuit, theta, derivatives):
    """(1 + P, 2^n) rows psi, d_0 psi .. d_{P-1} psi (only psi without derivatives)."""
    n, P = circuit.n, circuit.num_params
    masks = circuit.gate_masks()
    S = torch.zeros((1 + (P if derivatives else 0), 1 << n), dtype=torch.complex128, device=_dev())
    S[0, 0] = 1
    live = 1
    for (kind, q0, q1, param), m in zip(circuit.gates.tolist(), masks):
        if param < 0:
            _fixed(S[:live], n, kind, q0, q1)
            continue
        _rotate(S[:live], n, kind, q0, q1, m, float(theta[param]))
        if derivatives:  # dU psi = (-i/2) K U psi
            S[live:live + 1] = _generator(S[:1], n, kind, q0, q1, m) * -0.5j
            live += 1
    return S


def _hamiltonian(psi, n, ham):
    out = torch.zeros_like(psi)
    for c, x, z in zip(ham.coeffs, ham.xmask, ham.zmask):
        out += float(c) * _pauli_apply(psi, n, int(x), int(z))
    return out


def _one(p, theta, energy=True):
    S = _stack(p.circuit, theta, True)
    psi, D = S[:1], S[1:]
    G = torch.zeros((D.shape[0],) * 2, dtype=torch.complex128, device=S.device)
    step = max(1, (1 << 22) >> 2)
    for k in range(0, S.shape[1], step):  # slices of the states: no second copy of the stack
        d = D[:, k:k + step]
        G += d.conj() @ d.T
    t = (D @ psi[0].conj())  # <psi|d_j psi>
    G = G - t.conj()[:, None] * t[None, :]
    out = {"G": G, "t": t}
    if energy:
        h = _hamiltonian(psi, p.n, p.hamiltonian)
        out["energy"] = torch.real(torch.sum(psi.conj() * h)).reshape(1)
        out["grad"] = 2 * torch.real(D @ h[0].conj())
    return out


def exact(case, seed):
    problems = _problems(case, seed)
    call = case["call"]
    if call in ("metric", "qgt"):
        o = _one(problems[0], problems[0].theta, energy=False)
        if call == "qgt":
            return {"G": o["G"].reshape(-1)}
        # T_j = <psi|d_j psi> = -(i/2) <sigma_j>
        return {"g": o["G"].real.reshape(-1), "sigma": -2 * o["t"].imag}
    if call == "step":
        outs = [_one(p, p.theta) for p in problems]
        res = {"g": torch.cat([o["G"].real.reshape(-1) for o in outs]), "grad": torch.cat([o["grad"] for o in outs]),
               "energy": torch.cat([o["energy"] for o in outs]), "dtheta": None}
        if case["prec"] == "c128":
            res["dtheta"] = torch.cat([_solve(o) for o in outs])
        # complex64: dtheta is the solution of a system whose matrix and right-hand side carry float32
        # rounding, times its condition number; which side of the float64 solution it falls on says
        # nothing of the precision, so it is held by the tolerance alone and g and grad by this
        return res
    if call == "optimize":
        p = problems[0]
        theta = torch.as_tensor(p.theta, dtype=torch.float64, device=_dev()).clone()
        energies = []
        for _ in range(case["iters"]):
            o = _one(p, theta.cpu().numpy())
            energies.append(o["energy"])
            theta = theta + _solve(o)
        return {"theta": theta, "energies": torch.stack(energies)}
    p = problems[0]
    S = _stack(p.circuit, p.theta, True)
    h = _hamiltonian(S[:1], p.n, p.hamiltonian)
    return {"energy": torch.real(torch.sum(S[:1].conj() * h)).reshape(1), "grad": 2 * torch.real(S[1:] @ h[0].conj())}


def _solve(o):
    g = o["G"].real
    A = (g + LAM * torch.eye(g.shape[0], dtype=torch.float64, device=g.device)).cpu().numpy()
    return torch.as_tensor(np.linalg.solve(A, -DT * o["grad"].cpu().numpy()), device=g.device)
