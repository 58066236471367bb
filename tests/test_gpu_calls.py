"""mu_ex calls: the recorded graph of small grids against the launches it
replaces, and the checks of host calls.

Both forms run the same kernels on the same values, so results are equal bit
for bit; wide z kernels are compared with the oracle at the parity bar (1e-10).
"""
import numpy as np
import pytest

from oracle import oracle
from workloads import mu_microbench

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pnp():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1407_0674_gb300 import build, pnp as mod
    build.build()
    return mod


@pytest.mark.parametrize("precision", ["fp64", "df64", "fp32"])
@pytest.mark.parametrize("shape", [(12, 12, 12), (33, 9, 14)])
def test_graph_calls_equal_launches(pnp, precision, shape):
    import torch
    spec, rho = mu_microbench(shape=shape)
    ins = [torch.from_numpy(rho * f).cuda() for f in (1.0, 0.5, 0.9)]
    with pnp.Problem(spec, precision=precision) as P:
        want = []
        P.stage_timing(True)                  # timed calls are launched one by one
        for d in ins:
            out = torch.empty_like(d)
            P.excess_mu_device(d, out)
            assert P.status() == pnp.OK
            want.append(out.cpu().numpy())
        P.stage_timing(False)
        side = torch.cuda.Stream()
        for k in range(9):                    # fresh buffers, two streams
            d, out = ins[k % 3].clone(), torch.full_like(ins[0], np.nan)
            torch.cuda.synchronize()
            P.excess_mu_device(d, out, stream=side.cuda_stream if k % 2 else None)
            assert P.status() == pnp.OK
            assert np.array_equal(out.cpu().numpy(), want[k % 3])
        # a stream under capture records the launches
        d, out = ins[1].clone(), torch.zeros_like(ins[0])
        torch.cuda.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g):
            P.excess_mu_device(d, out, stream=torch.cuda.current_stream().cuda_stream)
        g.replay()
        torch.cuda.synchronize()
        assert np.array_equal(out.cpu().numpy(), want[1])


def test_host_call_checks_values(pnp):
    spec, rho = mu_microbench(10)
    with pnp.Problem(spec) as P:
        good = P.excess_mu(rho)
        for bad in (-1e-300, np.nan, np.inf):
            r = rho.copy()
            r[2, 9, 9, 9] = bad
            out = np.full_like(r, 7.0)
            rc = pnp.lib().pnp_excess_mu(P.h, pnp._ptr(r), pnp._ptr(out), -1)
            assert rc == pnp.ERR_INVALID and (out == 7.0).all()
            assert P.status() == pnp.OK
        assert np.array_equal(P.excess_mu(rho), good)
        zero = np.zeros_like(rho)
        zero[0, 0, 0, 0] = -0.0
        assert np.isfinite(P.excess_mu(zero)).all()


@pytest.mark.parametrize("species", [1, 3, 5])
@pytest.mark.parametrize("length", [16, 20, 24, 40, 48, 64, 80, 96])
def test_wide_z_kernels_match_oracle(pnp, length, species):
    spec, rho = mu_microbench(shape=(6, 7, length - 4))
    R, rb = (1.5, 2.0, 3.0, 1.0, 2.5)[:species], (0.004, 0.002, 0.0005, 0.004, 0.001)[:species]
    spec.R, spec.rho_b, spec.q, spec.depth = R, rb, (1, -1, 0, 1, -1)[:species], (0.0,) * species
    spec.fft_len = (16, 16, length)
    rng = np.random.default_rng(length + species)
    rho = np.stack([r * rng.lognormal(0.0, 0.1, spec.shape) for r in rb])
    ref, bad = oracle.excess_mu(spec, rho)
    assert bad == 0
    with pnp.Problem(spec) as P:
        for precision in ("fp64", "df64"):
            mu = P.excess_mu(rho, precision=precision)
            assert np.abs(mu - ref).max() <= 1e-10 * np.abs(ref).max()


@pytest.mark.parametrize("mode", ["global", "thread_local", "relaxed"])
def test_small_calls_beside_a_capture(pnp, mode):
    """Calls on one stream, the one that records the graph among them, leave a
    capture under way on another stream intact."""
    import torch
    spec, rho = mu_microbench(12)
    d = torch.from_numpy(rho).cuda()
    with pnp.Problem(spec) as P:
        want = torch.empty_like(d)
        P.excess_mu_device(d, want)               # buffers and spectra exist from here on
        assert P.status() == pnp.OK
        outs = [torch.full_like(d, np.nan) for _ in range(4)]
        x, side = torch.zeros(1000, device="cuda"), torch.cuda.Stream()
        torch.cuda.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, capture_error_mode=mode):
            x += 1
            for out in outs:
                P.excess_mu_device(d, out, stream=side.cuda_stream)
        g.replay()
        torch.cuda.synchronize()
        assert float(x[0]) == 1.0 and P.status() == pnp.OK
        assert all(torch.equal(out, want) for out in outs)


def test_small_calls_keep_their_stream_priority(pnp):
    """Calls on a high-priority stream finish while a kernel of many more blocks
    than the GPU holds is still running on another stream; at equal priority they would
    wait for its last block.  One call is on a stream of the default priority; those
    after it, on the first stream again, are still ahead."""
    import torch
    spec, rho = mu_microbench(12)
    d = torch.from_numpy(rho).cuda()
    big = torch.full((400_000_000,), 0.3, dtype=torch.float64, device="cuda")
    torch.sin_(big)                               # 13 ms of FP64 arithmetic, no library start-up below
    hi, low, work = torch.cuda.Stream(priority=-1), torch.cuda.Stream(), torch.cuda.Stream()
    with pnp.Problem(spec) as P:
        want, out = torch.empty_like(d), torch.empty_like(d)
        P.excess_mu_device(d, want)
        assert P.status() == pnp.OK
        for call, stream in enumerate([hi] * 6 + [low, hi, hi]):
            out.fill_(np.nan)
            torch.cuda.synchronize()
            done = torch.cuda.Event()
            with torch.cuda.stream(work):
                torch.sin_(big)
                done.record(work)
            P.excess_mu_device(d, out, stream=stream.cuda_stream)
            stream.synchronize()
            assert stream is low or not done.query(), call
            torch.cuda.synchronize()
            assert torch.equal(out, want)


@pytest.mark.parametrize("case,precision", [("wells", "fp64"), ("wells", "df64"), ("msa", "fp64"), ("msa", "fp32"),
                                            ("white bear", "fp64"), ("y 256", "tf32split")])
def test_graph_calls_of_every_option(pnp, case, precision):
    """The recorded graph takes each call's own buffers with every part of the pipeline on."""
    import torch
    from workloads import film_gummel, lognormal_density
    if case == "wells":
        spec = film_gummel(12, 10, 14, nsites=4)
        rho = lognormal_density(spec, 5, sigma=0.2)
    else:
        spec, rho = mu_microbench(shape=(12, 100, 9) if case == "y 256" else (12, 10, 9))
        spec.msa, spec.fmt = case == "msa", int(case == "white bear")
        if case == "y 256":
            spec.fft_len = (16, 256, 16)          # the length that the tensor-core y pass takes
    ins = [torch.from_numpy(rho * f).cuda() for f in (1.0, 0.5, 0.9)]
    with pnp.Problem(spec, precision=precision) as P:
        outs = [torch.full_like(ins[0], np.nan) for _ in range(7)]
        torch.cuda.synchronize()
        for k, out in enumerate(outs):
            P.excess_mu_device(ins[k % 3], out)
            assert P.status() == pnp.OK
        P.stage_timing(True)                      # timed calls are launched one by one
        for k, out in enumerate(outs):
            want = torch.full_like(out, np.nan)
            torch.cuda.synchronize()
            P.excess_mu_device(ins[k % 3], want)
            assert P.status() == pnp.OK
            assert torch.equal(out, want), k


@pytest.mark.parametrize("shape", [(10, 10, 10), (112, 112, 112)])
def test_refused_host_call_changes_nothing(pnp, shape):
    """Refused densities leave a pending device status, the output and the next result as
    they were, and are refused for what they are when memory runs out too.  After a call
    on another stream the verdict is waited for before anything else runs."""
    import torch
    spec, rho = mu_microbench(shape=shape)
    bad = rho.copy()
    bad[2, -1, -1, -1] = -1.0
    out = np.full_like(rho, 7.0)
    with pnp.Problem(spec, precision="fp32") as P:
        def refused():
            rc = pnp.lib().pnp_excess_mu(P.h, pnp._ptr(bad), pnp._ptr(out), -1)
            return rc == pnp.ERR_INVALID and (out == 7.0).all()
        pnp.lib().pnp_test_fail_alloc_at(1)
        try:
            assert refused()
        finally:
            pnp.lib().pnp_test_fail_alloc_at(0)
        d = torch.from_numpy(rho).cuda()
        d_mu, packed = torch.empty_like(d), 4.0 * d
        side = torch.cuda.Stream()
        for stream in (None, side.cuda_stream):
            torch.cuda.synchronize()
            P.excess_mu_device(packed, d_mu, stream=stream)      # n3 above 1
            torch.cuda.synchronize()
            assert refused() and P.status() == pnp.ERR_PACKING
            assert refused() and P.status() == pnp.OK
        P.excess_mu_device(d, d_mu)
        assert P.status() == pnp.OK
        assert np.array_equal(P.excess_mu(rho), d_mu.cpu().numpy())
