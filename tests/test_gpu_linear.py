"""Linear solves of the Gummel loop at the edges of their multigrid kernels:
two relaxed sweeps against the oracle on grids that end in each kind of coarsest
level, wrap odd extents, and give the dot products' slots more than one point.

Bar: both sides solve to a relative residual of 1e-13, so the iterates agree to
1e-8 as in the trajectory tests.
"""
import numpy as np
import pytest

from oracle import oracle
from workloads import ProblemSpec, bulk_density

pytestmark = pytest.mark.gpu
TOL = 1e-8


@pytest.mark.parametrize("bc,nx,ny,nz", [
    ("PPD", 2, 2, 6),        # one small level and a 2 x 2 x 2 coarsest one
    ("PPD", 8, 8, 8),        # one CTA holds every level
    ("PPD", 10, 9, 11),      # 1 x 1 x 11 coarsest level: two lanes a point, odd wraps
    ("PPD", 10, 9, 23),      # 1 x 1 x 23: one lane a point
    ("PPD", 10, 9, 53),      # 1 x 1 x 53: sweeps in shared memory
    ("NPD", 14, 15, 12),     # no-flux walls, an odd extent that does not wrap below
    ("PPD", 18, 45, 15),     # odd levels above the one-CTA tail
    ("PPD", 48, 50, 60),     # 144000 points: two points in some slots
])
def test_two_sweeps_match_oracle(bc, nx, ny, nz):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1407_0674_gb300 import build, pnp
    build.build()
    rng = np.random.default_rng(nx * ny + nz)
    rb = bulk_density(0.05, 1.0)
    spec = ProblemSpec(nx=nx, ny=ny, nz=nz, bc=tuple(bc), R=(1.0, 1.0), q=(1, -1), rho_b=(rb, rb),
                       rho_f=rng.normal(0, 0.01, (nz, ny, nx)), phi_lo=0.0, phi_hi=0.5, D=(1.0, 0.7),
                       lambda_phi=0.3, lambda_rho=0.3, tol=1e-30, max_iter=2, lin_tol=1e-13, screened_poisson=True)
    ref = oracle.gummel(spec)
    with pnp.Problem(spec) as P:
        phi, rho, st = P.gummel_solve(raise_on_error=False)
    assert st["iterations"] == ref["iters"] == 2
    assert np.abs(phi - ref["phi"]).max() <= TOL * max(np.abs(ref["phi"]).max(), 1.0)
    assert np.abs(rho - ref["rho"]).max() <= TOL * np.abs(ref["rho"]).max()
