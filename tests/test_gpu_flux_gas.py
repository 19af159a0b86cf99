"""The Gauss-point flux over the gas and the Mach number: its moments are
polynomials in the degrees of freedom N = 2 / (gamma - 1) and its half-space
integrals run over an edge at -U / sqrt(p / rho), so both ends of each range
are compared with the oracle."""
import numpy as np
import pytest

from tests.gpu_util import dev, host, needs_gpu

pytestmark = [pytest.mark.gpu, needs_gpu]


def _pairs(rng, n, mach, gamma):
    """State pairs that differ by a few percent, normal Mach number up to +-mach."""
    rho, p = rng.uniform(0.7, 1.3, n), rng.uniform(0.7, 1.3, n)
    c = np.sqrt(gamma * p / rho)
    u, v = c * mach * rng.uniform(-1.0, 1.0, n), c * 0.5 * rng.uniform(-1.0, 1.0, n)
    out = []
    for _ in range(2):
        f = 1.0 + 0.02 * rng.uniform(-1.0, 1.0, (4, n))
        r, a, b, q = rho * f[0], u * f[1], v * f[2], p * f[3]
        w = np.zeros((n, 6, 4))
        w[:, 0] = np.stack([r, r * a, r * b, q / (gamma - 1.0) + 0.5 * r * (a * a + b * b)], 1)
        w[:, 1:] = 0.5 * rng.uniform(-1.0, 1.0, (n, 5, 4))
        out.append(np.ascontiguousarray(w))
    return out


@pytest.mark.parametrize("kinetic", [0, 1])
@pytest.mark.parametrize("gamma", [1.1, 1.4, 5.0 / 3.0, 2.0])
@pytest.mark.parametrize("mach,mu,prandtl", [(0.05, 1e-3, 1.0), (2.5, 0.0, 1.0), (2.5, 1e-3, 0.72)])
def test_point_flux_over_gas_and_mach(mach, mu, prandtl, gamma, kinetic):
    """FP64 within 1e-11 of each flux scale: some 2,000 roundings of 1.1e-16 on
    terms up to (1 + M^2) N / 2 ~ 70 times the flux (gamma = 1.1, Mach 2.5)."""
    from oracle import oracle as O
    from paper_1802_00704_gb300 import gks as G
    n, dt = 65, 0.004
    wl, wr = _pairs(np.random.default_rng(31), n, mach, gamma)
    kw = dict(gamma=gamma, mu=mu, prandtl=prandtl, slope0_mode=kinetic)
    got = host(G.point_flux(dev(wl), dev(wr), dt, **kw))
    ref = np.stack([O.point_flux(wl[q], wr[q], dt, **kw)[0] for q in range(n)])
    scale = np.max(np.abs(ref), axis=0)
    err = np.max(np.abs(got - ref), axis=0) / scale
    assert np.all(err <= 1e-11), err
