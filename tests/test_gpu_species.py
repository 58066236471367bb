"""Gummel sweeps with one, three and four species against the oracle.

An iteration solves the species' Nernst-Planck systems side by side on lanes, one of
them in the problem's own memory and the others in the mu_ex workspace as far as
they fit; species i runs on lane i modulo their number, so a lane's operators
and control record serve several species in turn.  Bar and inputs as in the
tests of the linear solves: both sides solve to a relative residual of 1e-13 and
agree to 1e-8.
"""
import numpy as np
import pytest

from oracle import oracle
from workloads import ProblemSpec, bulk_density

pytestmark = pytest.mark.gpu
TOL = 1e-8


@pytest.mark.parametrize("bc,nx,ny,nz,species", [
    ("PPD", 12, 12, 12, 1),     # one lane, nothing beside it
    ("PPD", 12, 10, 14, 3),     # two lanes: species 0 and 2 in turn
    ("PPD", 10, 9, 11, 4),      # two lanes, two species each, odd wraps
    ("NND", 8, 8, 10, 4),       # three lanes: species 0 and 3 in turn
    ("NPD", 15, 16, 12, 3),     # a lane for each
    ("PPD", 2, 2, 6, 3),        # no lane fits beside the first: all in turn
])
def test_species_on_lanes_match_oracle(bc, nx, ny, nz, species):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1407_0674_gb300 import build, pnp
    build.build()
    rng = np.random.default_rng(nx * ny * nz + species)
    rb = bulk_density(0.03, 1.0)
    spec = ProblemSpec(nx=nx, ny=ny, nz=nz, bc=tuple(bc), R=(1.0,) * species, q=(1, -1, 2, 0)[:species],
                       rho_b=(rb, 0.8 * rb, 0.5 * rb, 0.6 * rb)[:species],
                       rho_f=rng.normal(0, 0.01, (nz, ny, nx)), phi_lo=0.0, phi_hi=0.5,
                       D=(1.0, 0.7, 0.4, 2.0)[:species], lambda_phi=0.3, lambda_rho=0.3, tol=1e-30, max_iter=3,
                       lin_tol=1e-13, screened_poisson=True)
    ref = oracle.gummel(spec)
    with pnp.Problem(spec) as P:
        phi, rho, st = P.gummel_solve(raise_on_error=False)
        again = P.gummel_solve(raise_on_error=False)
    assert st["iterations"] == ref["iters"] == 3
    assert np.abs(phi - ref["phi"]).max() <= TOL * max(np.abs(ref["phi"]).max(), 1.0)
    for i in range(species):
        assert np.abs(rho[i] - ref["rho"][i]).max() <= TOL * np.abs(ref["rho"][i]).max()
    assert np.array_equal(phi, again[0]) and np.array_equal(rho, again[1])
