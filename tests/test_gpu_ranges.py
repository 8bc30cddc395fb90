"""Inputs at the ends of what the entry points take: Hamiltonian coefficients near the ends of float64's range, more
parameters than a launch grid's y dimension has tiles of the metric, more runs than it has blocks; and circuits on both sides of where a launch shape or a kernel changes."""
import numpy as np
import pytest
import torch

from paper_2011_02991_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def qng():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2011_02991_gb300 import build as B
    B.build()
    from paper_2011_02991_gb300 import qng as Q
    return Q


@pytest.mark.parametrize("scale", [1e-290, 1e-200, 1e-160, 1e160, 1e250, 1e300])
@pytest.mark.parametrize("n,path", [(5, 1), (13, 2)])
def test_hamiltonian_scale(qng, n, path, scale):
    """<E> and its gradient are linear in H: coefficients whose squares leave float64's range give the scaled
    result of ordinary ones, to the rounding of the scaling (2^-53 of each coefficient) and of complex128."""
    rng = np.random.Generator(np.random.PCG64([n, path]))
    c = W.layered_ansatz(n, 2)
    h = W.random_pauli_hamiltonian(n, 8, rng)
    theta = W.uniform_theta(c.num_params, rng)
    out = []
    for s in (1.0, scale):
        p = W.Problem("scaled", c, W.Hamiltonian(h.coeffs * s, h.xmask, h.zmask), theta, precision=W.C128)
        ctx = qng.Context(p, path=path)
        grad, energy = ctx.gradient(ctx.theta0())
        ctx.sync()
        out.append((grad.cpu().numpy() / s, float(energy[0]) / s))
    assert np.abs(out[1][0] - out[0][0]).max() <= 1e-12 * np.abs(out[0][0]).max()
    assert abs(out[1][1] - out[0][1]) <= 1e-12 * np.abs(h.coeffs).sum()


def test_metric_of_many_parameters(qng):
    """P = 11 617 on 17 qubits, an RY on each and then RZ on one after the other: 66 066 tiles of the metric. RY
    entries are 1/4 on the diagonal, RZ ones <Z_a Z_b> - <Z_a><Z_b> over 4 (a product state: sin^2 / 4 on one
    qubit), and the real part of <Y_a Z_b> vanishes."""
    n, P = 17, 11617
    rows = [[W.RY, q, -1, q] for q in range(n)] + [[W.RZ, k % n, -1, k] for k in range(n, P)]
    rng = np.random.Generator(np.random.PCG64(5))
    theta = W.uniform_theta(P, rng)
    p = W.Problem("many", W.Circuit(n, np.array(rows, dtype=np.int32)), W.tfim_chain(n, 1.0, 0.5), theta, precision=W.C64)
    ctx = qng.Context(p)
    g = ctx.metric(ctx.theta0()).view(P, P)
    ctx.sync()
    q = torch.arange(n, P, device=g.device) % n
    s2 = 0.25 * torch.sin(torch.as_tensor(theta[:n], device=g.device)) ** 2
    ref = torch.zeros_like(g)
    ref[:n, :n] = 0.25 * torch.eye(n, dtype=g.dtype, device=g.device)
    ref[n:, n:] = torch.where(q[:, None] == q[None, :], s2[q][:, None], torch.zeros((), dtype=g.dtype, device=g.device))
    assert float((g - ref).abs().max()) <= 1e-6


def test_streaming_many_runs(qng):
    """70 000 runs (a CZ between Hadamards each) on the streaming path, against the on-chip path's <E>."""
    n, runs = 13, 70000
    rows = [[W.RY, q, -1, q] for q in range(n)]
    for k in range(runs):
        rows += [[W.H, 0, -1, -1], [W.CZ, 0, 1 + k % (n - 1), -1]]
    rng = np.random.Generator(np.random.PCG64(6))
    p = W.Problem("runs", W.Circuit(n, np.array(rows, dtype=np.int32)), W.random_pauli_hamiltonian(n, 10, rng),
                  W.uniform_theta(n, rng), precision=W.C64)
    e = []
    for path in (1, 2):
        ctx = qng.Context(p, path=path)
        v = ctx.energy(ctx.theta0())
        ctx.sync()
        e.append(float(v[0]))
        ctx.close()
    assert abs(e[0] - e[1]) <= 2e-4 * np.abs(p.hamiltonian.coeffs).sum()


@pytest.mark.parametrize("n,path", [(9, 1), (13, 2)])
def test_norm_is_kept(qng, n, path):
    """H = 1: <E> is the state's squared norm after 80 layers, 80 n rotations and as many transitions with an odd
    number of Hadamards. Factors are unitary to 2^-61 each, so what is left is the float64 sum of <E>."""
    c = W.layered_ansatz(n, 40)
    zero = np.zeros(1, dtype=np.uint64)
    rng = np.random.Generator(np.random.PCG64(n))
    p = W.Problem("norm", c, W.Hamiltonian(np.ones(1), zero, zero), W.uniform_theta(c.num_params, rng), precision=W.C128)
    ctx = qng.Context(p, path=path)
    e = ctx.energy(ctx.theta0())
    ctx.sync()
    assert abs(float(e[0]) - 1.0) <= 2e-15


@pytest.mark.parametrize("n,path", [(14, 1), (20, 2)])
def test_vanishing_imaginary_part(qng, n, path):
    """RY and CZ keep the state real, so Im G = 0, and what is left of it is rounding, of which a quarter counts: of
    the inner products to multiples of 2^-62, uniform within one unit (deviation 0.29), one per amplitude on chip and
    one per warp of 512 amplitudes streaming, and of the vectors, a dozen of 2^-60 or 2^-58 an amplitude, which a unit
    vector sums to about that unit."""
    c = W.layered_ansatz(n, 2, (W.RY,), W.CZ)
    rng = np.random.Generator(np.random.PCG64(n))
    p = W.Problem("real", c, W.tfim_chain(n, 1.0, 0.5), W.uniform_theta(c.num_params, rng), precision=W.C128)
    ctx = qng.Context(p, path=path)
    G = ctx.metric_complex(ctx.theta0())
    ctx.sync()
    rms = float((G.imag ** 2).mean().sqrt())
    sums = 0.29 * 2.0 ** -62 * np.sqrt(2.0 ** n / (512 if path == 2 else 1))
    assert rms <= 1.5 * 0.25 * (sums + 2.0 ** (-58 if path == 2 else -60))


def _layered(n, layers, kinds=(W.RY, W.RX), ent=W.CNOT):
    return lambda seed: W.layered_ansatz(n, layers, kinds, ent)


def _general(n, P):
    return lambda seed: W.general_problem(n, P, seed).circuit


def _random(n, gates):
    return lambda seed: W.random_circuit(n, gates, np.random.Generator(np.random.PCG64([n, seed])))


SHAPES = {
    # gate by gate, or frames, by steps per parameter; one to eight qubits
    "tiny": [_layered(1, 4), _layered(2, 5), _layered(3, 3), _random(4, 40)],
    "small_frames": [_layered(2, 4, (W.RY, W.RZ), W.CZ), _layered(3, 3, (W.RY, W.RZ), W.CZ), _layered(7, 2, (W.RY, W.RZ), W.CZ)],
    "small_general": [_general(3 + k % 6, 20 + k) for k in range(10)],
    # 8 and 16 amplitudes a thread, CTAs of 64 to 512 threads, few instances and more
    "general": [_general(5 + k, 24) for k in range(8)],
    "general_more": [_general(4 + k, 20) for k in range(9)],
    "ten": [_layered(10, 2, (W.RY, W.RZ), W.CZ), _layered(6, 3)],
    "eleven": [_layered(11, 1, (W.RY, W.RZ), W.CZ), _random(5, 60)] + [_layered(4, 2)] * 7,
    "thirteen": [_layered(13, 1), _layered(9, 2)],
    "thirteen_general": [_general(13, 12)] + [_general(4 + k, 15) for k in range(8)],
    "thirteen_more": [_layered(13, 1)] + [_layered(3 + k, 2) for k in range(8)],
    # clusters of 8 CTAs
    "one13": [_layered(13, 1)],
    "one14": [_random(14, 40)],
    "one14_general": [_general(14, 14)],
    "one15": [_layered(15, 1, (W.RY, W.RZ), W.CZ)],
    "one15_general": [_general(15, 9)],
}


@pytest.mark.parametrize("precision", [W.C64, W.C128])
@pytest.mark.parametrize("name", sorted(SHAPES))
def test_shapes(qng, oracle, name, precision):
    """Metric, its imaginary part, gradient and energy of every instance against the oracle."""
    probs = []
    for k, make in enumerate(SHAPES[name]):
        c = make(300 + k)
        rng = np.random.Generator(np.random.PCG64([c.n, k]))
        probs.append(W.Problem(name, c, W.random_pauli_hamiltonian(c.n, 6, rng), W.uniform_theta(c.num_params, rng), precision=precision))
    ctx = qng.Context(probs if len(probs) > 1 else probs[0])
    G = ctx.metric_complex(ctx.theta0())
    g = ctx.metric(ctx.theta0())
    grad, e = ctx.gradient(ctx.theta0())
    ctx.sync()
    tol = 1e-10 if precision == W.C128 else 2e-4
    assert float((G.real - g).abs().max()) <= tol
    for p, Gp, gr, en in zip(probs, ctx.split_metric(G), ctx.split_params(grad), e.cpu().numpy()):
        ref = oracle.qng_step(p)
        scale = np.abs(p.hamiltonian.coeffs).sum()
        assert np.abs(Gp.cpu().numpy() - ref["G"]).max() <= tol / 4, p.n
        assert np.abs(gr.cpu().numpy() - ref["grad"]).max() <= tol * scale, p.n
        assert abs(en - ref["E"]) <= tol * scale, p.n
