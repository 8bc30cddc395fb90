"""Host checks of the diagonal-frame planner (no GPU): the program that the on-chip kernels run is
executed in float64 by a host-only probe (tests/frames_probe.cu, linking the library's planner) and
compared with the oracle: metric, its imaginary part, <sigma_j>, control probabilities, gradient and
energy. Circuits of every gate kind in every order, so that frames of every kind meet rotations,
CNOT networks, controlled and string rotations; 1 to 9 qubits, one to eight CTAs per vector."""
import itertools
import shutil
import subprocess

import numpy as np
import pytest

from paper_2011_02991_gb300 import workloads as W

ROOT = __import__("pathlib").Path(__file__).resolve().parents[1]


@pytest.fixture(scope="module")
def probe(tmp_path_factory):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not shutil.which(nvcc):
        pytest.skip("nvcc not found")
    exe = tmp_path_factory.mktemp("probe") / "frames_probe"
    src = ROOT / "paper_2011_02991_gb300" / "csrc"
    r = subprocess.run([nvcc, "-std=c++17", "-O1", "-I", str(ROOT / "include"), "-I", str(src), "-o", str(exe),
                        str(ROOT / "tests" / "frames_probe.cu"), str(src / "qng_frames_plan.cu")],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    return exe


def run_probe(exe, p, kb=4, cl=0, tb=0, low=0):
    c, h = p.circuit, p.hamiltonian
    lines = [f"{c.n} {c.num_params} {len(c.gates)} {h.num_terms} {kb} {cl} {tb} {low}"]
    for row, m in zip(c.gates, c.gate_masks()):
        lines.append(" ".join(str(int(v)) for v in row) + f" {int(m[0])} {int(m[1])}")
    lines += [f"{float(a)!r} {int(x)} {int(z)}" for a, x, z in zip(h.coeffs, h.xmask, h.zmask)]
    lines += [repr(float(t)) for t in p.theta]
    r = subprocess.run([str(exe)], input="\n".join(lines) + "\n", capture_output=True, text=True)
    out = r.stdout.strip().split("\n")
    assert r.returncode == 0 and out[-1] == "ok", f"probe: {out[-3:]} {r.stderr}"
    return {x.split()[0]: np.array([float(v) for v in x.split()[1:]]) for x in out if " " in x or x in ("L", "grad")}


def check(exe, oracle, p, kb=4, cl=0, tb=0, low=0):
    d = run_probe(exe, p, kb, cl, tb, low)
    ref = oracle.qng_step(p)
    P = p.P
    tol = 1e-11
    assert abs(d["E"][0] - ref["E"]) <= tol * max(1.0, np.abs(p.hamiltonian.coeffs).sum())
    if P == 0:
        return d
    assert np.abs(d["grad"] - ref["grad"]).max() <= tol * max(1.0, np.abs(p.hamiltonian.coeffs).sum())
    assert np.abs(d["sigma"] + 2 * ref["T"].imag).max() <= tol
    g = np.zeros((P, P), dtype=complex)
    iu = [(i, j) for j in range(P) for i in range(j)]
    for (i, j), v in zip(iu, d["L"].reshape(-1, 2)):
        g[i, j] = complex(v[0], v[1]) - 0.25 * d["sigma"][i] * d["sigma"][j]
        g[j, i] = np.conj(g[i, j])
    for j in range(P):
        g[j, j] = 0.25 * (d["ctrl"][j] - d["sigma"][j] ** 2)
    assert np.abs(g - ref["G"]).max() <= tol
    return d


@pytest.mark.parametrize("kb", [3, 4])
@pytest.mark.parametrize("seed", range(18))
def test_random_circuits(probe, oracle, seed, kb):
    """Every simple gate kind at random places, 1 to 9 qubits, 8 and 16 amplitudes per thread."""
    check(probe, oracle, W.random_problem(1 + seed % 9, 70, 6, 4000 + seed), kb)


@pytest.mark.parametrize("seed", range(8))
def test_generalised(probe, oracle, seed):
    """Controlled and Pauli-string rotations in frames of every kind."""
    check(probe, oracle, W.general_problem(3 + seed % 5, 50, 90 + seed), 3 + seed % 2)


@pytest.mark.parametrize("cl", [0, 1, 2, 3])
@pytest.mark.parametrize("kinds,ent", [((W.RY, W.RZ), W.CZ), ((W.RY, W.RX, W.RZ), W.CNOT), ((W.RX, W.RY), W.CNOT)])
def test_layered(probe, oracle, kinds, ent, cl):
    """Layered ansätze; every layer's rotations of one axis are one run."""
    n = 7
    c = W.layered_ansatz(n, 3, kinds, ent)
    rng = np.random.Generator(np.random.PCG64(3))
    p = W.Problem("l", c, W.random_pauli_hamiltonian(n, 9, rng), W.uniform_theta(c.num_params, rng))
    d = check(probe, oracle, p, 4, cl)
    check(probe, oracle, p, 3, cl)
    if kinds[-1] == W.RZ:
        assert d["runs"][0] <= 3 * len(kinds) + 1


@pytest.mark.parametrize("ent", [W.CZ, W.CNOT])
@pytest.mark.parametrize("kinds", [k for m in (1, 2, 3) for k in itertools.permutations((W.RX, W.RY, W.RZ), m)])
def test_runs_per_layer(probe, oracle, kinds, ent):
    """A layer costs one run per axis and at most one more, for the entangler's signs or S phases: a ladder is one
    transition, whatever rotations it follows."""
    n, layers = 6, 3
    c = W.layered_ansatz(n, layers, kinds, ent)
    rng = np.random.Generator(np.random.PCG64(5))
    p = W.Problem("l", c, W.random_pauli_hamiltonian(n, 9, rng), W.uniform_theta(c.num_params, rng))
    d = check(probe, oracle, p, 3)
    assert d["runs"][0] <= layers * (len(kinds) + 1) + 1
    check(probe, oracle, p, 3, 0, 5, 2)


def test_z_runs_and_no_parameters(probe, oracle):
    check(probe, oracle, W.z_run_problem(6, 80, 3))
    c = W.Circuit(3, np.array([[W.H, 0, -1, -1], [W.CNOT, 0, 2, -1], [W.Y, 1, -1, -1], [W.CZ, 0, 1, -1]], dtype=np.int32))
    h = W.hamiltonian_from_terms([(0.5, {0: "X", 2: "X"}), (0.25, {1: "Z"}), (-1.5, {0: "Y", 2: "Y"})])
    check(probe, oracle, W.Problem("fixed", c, h, np.zeros(0)))


def brickwork(n, layers, seed=0):
    """Layers of H on the even qubits and a CNOT from each to its neighbour, then one layer of RY: all of the Hadamards lie
    in one transition (the frame does not absorb one behind a CNOT)."""
    rows = []
    for k in range(layers):
        rows += [[W.H, q, -1, -1] for q in range(0, n, 2)] + [[W.CNOT, q, q + 1, -1] for q in range(0, n - 1, 2)]
    rows += [[W.RY, q, -1, q] for q in range(n)]
    rng = np.random.Generator(np.random.PCG64([n, layers, seed]))
    return W.Problem("brickwork", W.Circuit(n, np.array(rows, dtype=np.int32)), W.random_pauli_hamiltonian(n, 12, rng),
                     W.uniform_theta(n, rng))


@pytest.mark.parametrize("n,layers", [(5, 3), (6, 16), (7, 30), (9, 60)])
def test_long_transitions(probe, oracle, n, layers):
    """More Hadamards in one transition than a factor table can normalise (its entries are multiples of 2^-61)."""
    p = brickwork(n, layers)
    check(probe, oracle, p, 3)
    check(probe, oracle, p, 3, 0, 5, 2)


@pytest.mark.parametrize("n,kb,tb,low", [(7, 3, 5, 2), (9, 3, 6, 3)])
def test_stretch_with_a_sign(probe, oracle, n, kb, tb, low):
    """A stretch of CNOTs that begins with one that is a sign in its frame: the qubit that this one alone touches gets
    no Hadamard for the others, which a pass would meet next to a later one. (What a transition's Hadamards leave of
    the norm is what the run after it takes, whichever of them a pass executes together.)"""
    for top in (n - 1, n - 2, 3):
        rows, k = [], 0
        for kind in (W.RY, W.RZ):
            rows += [[kind, q, -1, k + q] for q in range(n)]
            k += n
        rows += [[W.H, 1, -1, -1], [W.H, 2, -1, -1], [W.CNOT, top, 1, -1], [W.CNOT, 2, top, -1], [W.H, 1, -1, -1], [W.CNOT, 1, 0, -1]]
        rows += [[W.RY, q, -1, k + q] for q in range(n)]
        rng = np.random.Generator(np.random.PCG64(n))
        p = W.Problem("sign", W.Circuit(n, np.array(rows, dtype=np.int32)), W.random_pauli_hamiltonian(n, 6, rng),
                      W.uniform_theta(k + n, rng))
        check(probe, oracle, p, kb)
        check(probe, oracle, p, kb, 0, tb, low)


@pytest.mark.parametrize("n,kb,tb,low", [(7, 3, 5, 2), (9, 3, 6, 3), (8, 3, 7, 3), (9, 4, 6, 1), (10, 3, 6, 3), (6, 4, 6, 2)])
@pytest.mark.parametrize("seed", range(4))
def test_streaming_passes(probe, oracle, n, kb, tb, low, seed):
    """Passes over tiles: one to four windows over the index bits, CNOTs whose control lies outside the
    tile, runs that start in the middle of a pass."""
    check(probe, oracle, W.random_problem(n, 60, 6, 5000 + seed), kb, 0, tb, low)


@pytest.mark.parametrize("kinds,ent", [((W.RY, W.RZ), W.CZ), ((W.RY, W.RX, W.RZ), W.CNOT)])
def test_streaming_layered(probe, oracle, kinds, ent):
    """Two windows over the index bits: one pass per run, and one more per CNOT ladder."""
    n = 9
    c = W.layered_ansatz(n, 2, kinds, ent)
    rng = np.random.Generator(np.random.PCG64(4))
    p = W.Problem("l", c, W.random_pauli_hamiltonian(n, 9, rng), W.uniform_theta(c.num_params, rng))
    d = check(probe, oracle, p, 3, 0, 6, 3)
    assert d["passes"][1] <= d["runs"][0] + (2 if ent == W.CNOT else 0)
    fixed = W.Circuit(6, np.array([[W.H, 0, -1, -1], [W.Z, 2, -1, -1]], dtype=np.int32))
    check(probe, oracle, W.Problem("fixed", fixed, W.tfim_chain(6, 1.0, 0.3), np.zeros(0)), 3, 0, 5, 2)
