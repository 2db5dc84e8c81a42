"""The FP64 sweeps' state between launches: runs split off a refresh, non-finite matrices, and what one
measurement adds."""
import math

import numpy as np
import pytest

from paper_1006_2716_gb300 import workloads as wl

pytestmark = pytest.mark.gpu

LS = [8, 12, 16, 20, 24, 32, 40, 48, 64]


@pytest.fixture(scope="module")
def hf():
    import torch

    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    from paper_1006_2716_gb300 import build as B

    B.build()
    from paper_1006_2716_gb300 import hf as H

    return H


def _context(hf, L, U, n=6, cps=4, bin_size=2):
    cfg = dict(wl.CONFIGS["square6"], Lx=n, Ly=n, beta=0.25 * L, dtau=0.25, U=U, chains_per_site=cps,
               refresh_every=10, bin_size=bin_size, max_bins=4, n_matsubara=4, seed=17)
    ctx = hf.Context(hf.make_params(cfg))
    baths = wl.random_baths(3 * L, ctx.n_sites, 0.25 * L, L)
    for i in range(ctx.n_sites):
        for sp in range(2):
            hf.hf_set_g0(ctx.handle, i, sp, baths[i, sp])
    return ctx


def _state(hf, ctx):
    hf.hf_sync(ctx.handle)
    G = np.array([hf.hf_get_green(ctx.handle, c, ctx.L) for c in range(ctx.n_chains)])
    obs = [hf.hf_measure(ctx.handle, i, ctx.L) for i in range(ctx.n_sites)]
    fields, count = hf.hf_get_fields(ctx.handle, ctx.n_chains, ctx.L)
    acc = hf.hf_get_accepts(ctx.handle, ctx.n_chains)
    return [G, fields, count, acc] + [np.concatenate([np.ravel(x) for x in ob]) for ob in obs]


@pytest.mark.parametrize("U", [0.0, 8.0, 16.0])      # 16: updates in FP64 arithmetic
@pytest.mark.parametrize("L", LS)
def test_a_run_in_several_launches_is_the_run_in_one(hf, L, U):
    """Split off the refreshes (after sweeps 10, 20 of a chain) and within a bin: bit for bit."""
    out = []
    for launches in (((15, 8),), ((7, 0), (8, 3), (0, 5)), ((13, 0), (1, 0), (1, 1), (0, 7))):
        ctx = _context(hf, L, U)
        for k, (w, m) in enumerate(launches):
            hf.hf_sweep(ctx.handle, w, m, 1 if k == 0 else 0)
        out.append(_state(hf, ctx))
        ctx.close()
    for other in out[1:]:
        assert all(np.array_equal(a, b) for a, b in zip(out[0], other))


@pytest.mark.parametrize("L", [8, 32, 40, 64])
def test_a_matrix_that_is_not_finite_stays_so(hf, L):
    """A zero bath has no inverse: the launch reports it, a further launch without a refresh reports it
    again, and the matrix and the observables of that spin show it until a refresh finds a good
    bath."""
    ctx = _context(hf, L, 8.0, n=1, cps=2)
    good = hf.hf_get_g0(ctx.handle, 1, L)[0]
    hf.hf_set_g0(ctx.handle, 0, 1, np.zeros(L))
    for k in range(3):
        hf.hf_sweep(ctx.handle, 0, 4 if k else 0, 1 if k == 0 else 0)
        with pytest.raises(hf.HFError) as e:
            hf.hf_sync(ctx.handle)
        assert e.value.status == hf.HF_ENUMERIC
        G = hf.hf_get_green(ctx.handle, 0, L)
        assert np.all(np.isfinite(G[0])) and not np.any(np.isfinite(G[1]))
    gtau, n, d, m, _ = hf.hf_measure(ctx.handle, 0, L)
    assert np.all(np.isfinite(gtau[:L])) and np.all(np.isnan(gtau[L:]))
    assert np.isfinite(n[0]) and np.isnan(n[1]) and np.isnan(d) and np.isnan(m)
    assert not hf.hf_get_accepts(ctx.handle, 2).any()
    hf.hf_set_g0(ctx.handle, 0, 1, good[1])
    hf.hf_clear_measurements(ctx.handle)
    hf.hf_sweep(ctx.handle, 0, 4, 1)
    assert all(np.all(np.isfinite(x)) for x in _state(hf, ctx))
    ctx.close()


@pytest.mark.parametrize("L,U", [(16, 12.0), (32, 12.0), (40, 8.0), (64, 12.0)])
def test_a_measurement_is_the_sum_over_g(hf, L, U):
    """One measurement against the exact sums over the stored G: every element of that is rounded to
    2^-53 of itself, and so are the result and the sums behind n."""
    ctx = _context(hf, L, U, n=14, cps=1, bin_size=1)
    hf.hf_sweep(ctx.handle, 7, 1, 1)
    for i in range(ctx.n_sites):
        got = hf.hf_measure(ctx.handle, i, L)[0]
        G = hf.hf_get_green(ctx.handle, i, L)
        for sp in range(2):
            for m in range(L):
                x = [(1.0 if l + m < L else -1.0) * G[sp, (l + m) % L, l] for l in range(L)]
                tol = 4 * 2.0 ** -53 * math.fsum(map(abs, x)) / L
                assert abs(got[sp * L + m] - math.fsum(x) / L) <= tol, (i, sp, m)
    ctx.close()


def test_a_batch_of_both_updates_is_its_problems_alone(hf):
    """Rows of 57 and 59 bits, L = 64 and FP64 updates (dtau U > 3) in one captured iteration: every
    problem's state and self-energy are those of its own iterations, bit for bit."""
    import torch

    stream = torch.cuda.Stream()
    problems = [(16, 2.0), (32, 8.0), (64, 8.0), (20, 16.0), (64, 14.0)]
    alone, fused = [], []
    for group in (alone, fused):
        for k, (L, U) in enumerate(problems):
            cfg = dict(wl.CONFIGS["square6"], beta=0.25 * L, dtau=0.25, U=U, mu=U / 2, chains_per_site=3,
                       n_warmup=4, n_measure=12, bin_size=4, max_bins=3, refresh_every=5, n_matsubara=64,
                       seed=70 + k)
            group.append(hf.Context(hf.make_params(cfg), stream=stream))
    batch = hf.hf_batch_create([c.handle for c in fused], 1)
    for _ in range(3):
        hf.hf_batch_rdmft_step(batch)
        for c in alone:
            hf.hf_rdmft_step(c.handle)
    for a, f in zip(alone, fused):
        assert all(np.array_equal(x, y) for x, y in zip(_state(hf, a), _state(hf, f)))
        assert np.array_equal(hf.hf_get_sigma(a.handle, a.n_sites, 64), hf.hf_get_sigma(f.handle, f.n_sites, 64))
    hf.hf_batch_free(batch)
    for c in alone + fused:
        c.close()


def test_served_solves_of_both_updates_share_a_launch(hf):
    """The same request alone and among others of either form gives the same result."""
    def server():
        p = hf.hf_srv_params()
        for k, v in dict(chains_per_request=4, n_warmup=6, n_measure=12, refresh_every=5, bin_size=4, precision=0,
                         team_warps=0, max_L=64, max_inflight=32, max_keys=64, n_streams=2,
                         requests_per_launch=16).items():
            setattr(p, k, v)
        return hf.Server(p)

    def request(k, L, U):
        return hf.make_request(0, k, L, 0.25 * L, U, 5, wl.random_baths(300 + k, 1, 0.25 * L, L)[0])

    mix = [request(k, L, U) for k, (L, U) in enumerate([(16, 2.0), (20, 16.0), (64, 8.0), (64, 14.0), (32, 8.0)] * 3)]
    s = server()
    tickets = [hf.hf_srv_submit(s.handle, r) for r in mix]
    together = [hf.hf_srv_wait(s.handle, t) for t in tickets]
    s.close()
    for r, want in zip(mix, together):
        s = server()
        got = hf.hf_srv_wait(s.handle, hf.hf_srv_submit(s.handle, r))
        s.close()
        for key in want:
            if "latency" not in key and "ticket" not in key:
                assert np.array_equal(np.asarray(want[key]), np.asarray(got[key])), key
