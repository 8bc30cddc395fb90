"""Inputs at the ends of what the entry points take: Hamiltonian coefficients near the ends of float64's range."""
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
