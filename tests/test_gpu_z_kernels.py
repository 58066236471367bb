"""z kernels of mu_ex on both sides of their dispatch against the oracle: the
paired-column form, which planes of many padded columns take, and the form with
ten thread groups a column, which small planes take.

The domain is a few points wide, so the oracle is quick; the padded lengths in x
and y alone decide which form runs.  Bars: those of the mu_ex parity tests (1e-10 in
FP64 and double-float, 2e-5 in FP32).
"""
import numpy as np
import pytest

from oracle import oracle
from workloads import mu_microbench

pytestmark = pytest.mark.gpu
TOL = {"fp64": 1e-10, "df64": 1e-10, "fp32": 2e-5}
RADII, BULK, CHARGE = (1.5, 2.0, 3.0, 1.0, 2.5), (0.004, 0.002, 0.0005, 0.004, 0.001), (1, -1, 0, 1, -1)


@pytest.fixture(scope="module")
def pnp():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1407_0674_gb300 import build, pnp as mod
    build.build()
    return mod


def check(pnp, plane, length, species, precisions):
    spec, _ = mu_microbench(shape=(6, 7, length - 4))
    spec.R, spec.rho_b, spec.q, spec.depth = RADII[:species], BULK[:species], CHARGE[:species], (0.0,) * species
    spec.fft_len = (*plane, length)
    rng = np.random.default_rng(100 * length + species)
    rho = np.stack([r * rng.lognormal(0.0, 0.1, spec.shape) for r in spec.rho_b])
    ref, bad = oracle.excess_mu(spec, rho)
    assert bad == 0
    with pnp.Problem(spec) as P:
        assert P.info()["fft_len"] == (*plane, length)
        for precision in precisions:
            mu = P.excess_mu(rho, precision=precision)
            for i in range(species):
                assert np.abs(mu[i] - ref[i]).max() <= TOL[precision] * np.abs(ref[i]).max(), precision


# 65 x 49 columns of (ky, Ly - ky) pairs: at least 796 warps in every form
@pytest.mark.parametrize("length,species", [(16, 3), (20, 3), (24, 1), (24, 3), (24, 5), (32, 3), (40, 3), (48, 3),
                                            (64, 3), (80, 1), (80, 3), (80, 5), (96, 3), (128, 3)])
def test_paired_column_kernels_match_oracle(pnp, length, species):
    check(pnp, (128, 96), length, species, ("fp64", "df64", "fp32"))


@pytest.mark.parametrize("length", [16, 20, 24, 32, 40, 48, 64, 80, 96, 128])
def test_small_planes_in_fp32_match_oracle(pnp, length):
    check(pnp, (16, 16), length, 3, ("fp32",))
    check(pnp, (40, 24), length, 4, ("fp32",))


# planes at the limits of the rule for the columns per CTA: rows of one sector, fewer
# on planes whose fullest SM empties by half, few large CTAs of 8-lane columns
@pytest.mark.parametrize("plane,length", [((64, 64), 48), ((40, 80), 48), ((32, 64), 80), ((32, 64), 96),
                                          ((90, 90), 40), ((64, 64), 64), ((64, 64), 40), ((32, 64), 128)])
def test_column_tiles_match_oracle(pnp, plane, length):
    check(pnp, plane, length, 3, ("fp64", "df64", "fp32"))


@pytest.mark.parametrize("length", [64, 96, 128])
def test_msa_column_tiles_match_oracle(pnp, length):
    """The z back with the MSA term keeps the paired-column form and a tile of its own."""
    spec, _ = mu_microbench(shape=(6, 7, length - 8))
    spec.msa, spec.fft_len = True, (40, 48, length)
    rng = np.random.default_rng(length)
    rho = np.stack([r * rng.lognormal(0.0, 0.1, spec.shape) for r in BULK[:3]])
    ref, bad = oracle.excess_mu(spec, rho)
    assert bad == 0
    with pnp.Problem(spec) as P:
        for precision in ("fp64", "df64", "fp32"):
            for _ in range(2):
                mu = P.excess_mu(rho, precision=precision)
                for i in range(3):
                    assert np.abs(mu[i] - ref[i]).max() <= TOL[precision] * np.abs(ref[i]).max(), precision
