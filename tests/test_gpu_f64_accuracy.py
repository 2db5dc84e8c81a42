"""Accuracy of the FP64 sweeps between two refreshes: after some sweeps of Sherman-Morrison
updates, G is compared with the same updates in 113-bit arithmetic (green_error.cpp), beside what
rank-1 updates in FP64 reach from the same matrices."""
import ctypes as C
import os
import subprocess

import numpy as np
import pytest

import oracle as o
from paper_1006_2716_gb300 import workloads as wl

pytestmark = pytest.mark.gpu

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def hf():
    import torch

    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    from paper_1006_2716_gb300 import build as B

    B.build()
    from paper_1006_2716_gb300 import hf as H

    return H


@pytest.fixture(scope="module")
def helper(tmp_path_factory):
    so = str(tmp_path_factory.mktemp("green") / "libgreen_error.so")
    subprocess.run(["g++", "-O2", "-std=c++17", "-ffp-contract=off", "-fPIC", "-shared", "-pthread",
                    "-o", so, os.path.join(HERE, "green_error.cpp")], check=True)
    return C.CDLL(so)


def sweep_errors(hf, helper, L, U, dtau, chains, nsweep):
    """[chains][2] errors of the library's G and of FP64 rank-1 updates after nsweep sweeps from a
    refreshed state (relative to max|G|), over one random bath per 8 chains."""
    beta, cps = L * dtau, 8
    err = np.zeros((chains, 2))
    err64 = np.zeros((chains, 2))
    _, lam = o.constants(beta, U, L)
    for c0 in range(0, chains, cps):
        cfg = dict(wl.CONFIGS["square6"], Lx=1, Ly=1, beta=beta, dtau=dtau, U=U, chains_per_site=cps,
                   refresh_every=1000, bin_size=4, max_bins=1, seed=99 + c0, n_matsubara=4)
        ctx = hf.Context(hf.make_params(cfg))
        bath = wl.random_baths(31 * L + c0, 1, beta, L)[0]
        for sp in range(2):
            hf.hf_set_g0(ctx.handle, 0, sp, bath[sp])
        hf.hf_sweep(ctx.handle, 10, 0, 1)
        hf.hf_sweep(ctx.handle, 0, 0, 1)
        s0, _ = hf.hf_get_fields(ctx.handle, cps, L)
        G0 = np.array([hf.hf_get_green(ctx.handle, c, L) for c in range(cps)])
        hf.hf_sweep(ctx.handle, nsweep, 0, 0)
        s1, _ = hf.hf_get_fields(ctx.handle, cps, L)
        G1 = np.array([hf.hf_get_green(ctx.handle, c, L) for c in range(cps)])
        ctx.close()
        u = np.array([[[o.uniform(cfg["seed"], 0, c, 10 + w, l) for l in range(L)]
                       for w in range(nsweep)] for c in range(cps)])
        e, e64, s = np.zeros((cps, 2)), np.zeros((cps, 2)), np.zeros((cps, L), dtype=np.int8)
        dp = lambda a: a.ctypes.data_as(C.POINTER(C.c_double))
        i8 = lambda a: a.ctypes.data_as(C.POINTER(C.c_int8))
        s0 = np.ascontiguousarray(s0, dtype=np.int8)
        helper.green_errors(L, cps, nsweep, C.c_double(np.exp(-2 * lam) - 1), C.c_double(np.exp(2 * lam) - 1),
                            dp(G0), i8(s0), dp(u), dp(G1), dp(e), dp(e64), i8(s))
        assert np.array_equal(s, s1)
        err[c0:c0 + cps], err64[c0:c0 + cps] = e, e64
    return err, err64


@pytest.mark.parametrize("L,U", [(8, 120.0), (16, 80.0), (20, 12.1), (24, 32.0), (64, 40.0)])
def test_strong_coupling_updates_are_fp64s(hf, helper, L, U):
    """dtau U > 3: G is as close to exact updates as FP64 rank-1 updates are.  The two sides round
    in a different order, and one interval's error scatters around the other's by the spread of
    single roundings, so the worst and the 90 % mark over 128 matrices agree within a factor of
    eight; 1e-15 for intervals without a flip."""
    err, err64 = sweep_errors(hf, helper, L, U, 0.25, 64, 10)
    for q in (0.9, 1.0):
        assert np.quantile(err, q) <= 8 * np.quantile(err64, q) + 1e-15, (q, np.quantile(err, q), np.quantile(err64, q))


@pytest.mark.parametrize("U", [8.0, 12.0])
@pytest.mark.parametrize("L", [8, 12, 16, 20, 24, 32, 40, 48, 64])
def test_usual_coupling_updates_are_no_worse_than_fp64s(hf, helper, L, U):
    """dtau U = 2 and 3: nine intervals of ten end no further from exact updates than FP64 rank-1
    updates from the same matrices do.  The 99 % mark is the sixth largest of 512 heavy-tailed errors
    and scatters by itself, so there a factor of three is allowed."""
    err, err64 = sweep_errors(hf, helper, L, U, 0.25, 256, 10)
    for q, f in ((0.5, 1.0), (0.9, 1.0), (0.99, 3.0)):
        assert np.quantile(err, q) <= f * np.quantile(err64, q) + 1e-15, (q, np.quantile(err, q), np.quantile(err64, q))


def near_singular_flip(L, U, dtau, R=1e-11):
    """(bath [2][L], fields, chain seed, slice): a chain whose first sweep accepts one flip only, with a
    ratio near R for spin up and near 1 / R for spin down.  A bath scaled by x has a singular Dyson
    matrix for given fields where 1/x is an eigenvalue of g0 (1 - e^-V); spin up is put there for the
    flipped fields, spin down for the present ones."""
    beta = L * dtau
    _, lam = o.constants(beta, U, L)
    rng = np.random.default_rng(5)
    d = np.arange(L)[:, None] - np.arange(L)[None]
    for seed in range(100000):
        bath = wl.random_baths(seed, 1, beta, L)[0].copy()
        s = rng.choice([-1, 1], L)
        at = int(rng.integers(L))
        G = []
        for sp, sg in ((0, 1), (1, -1)):
            f = s.copy()
            if sp == 0:
                f[at] = -f[at]
            sign = np.where(d >= 0, 1.0, -1.0)
            w = np.linalg.eigvals(sign * bath[sp][d % L] * (1 - np.exp(-sg * lam * f)))
            w = w[(np.abs(w.imag) < 1e-12 * np.abs(w)) & (w.real > 0)].real
            if not len(w):
                break
            bath[sp] *= (1 + R * rng.choice([-1, 1])) / w[np.argmin(np.abs(np.log(w)))]
            ev = np.exp(sg * lam * s)
            G.append(np.linalg.inv(np.linalg.inv(sign * bath[sp][d % L]) * ev - np.diag(ev - 1)))
        flips = []
        for l in range(L if len(G) == 2 else 0):
            a = [np.exp(-2 * lam * sg * s[l]) - 1 for sg in (1, -1)]
            r = [1 + (1 - G[sp][l, l]) * a[sp] for sp in (0, 1)]
            if o.uniform(seed, 0, 0, 0, l) < r[0] * r[1]:
                flips.append(l)
                G = [g + a[sp] / r[sp] * np.outer(g[:, l] - np.eye(L)[l], g[l]) for sp, g in enumerate(G)]
                if abs(r[0]) > 1e-9 or len(flips) > 1:
                    break
        else:
            if flips == [at]:
                return bath, s, seed, at
    raise AssertionError("no such chain found")


@pytest.mark.parametrize("L", [8, 12, 16])
def test_a_nearly_singular_flip_is_right(hf, helper, L):
    """A flip whose ratio is R = 1e-11 to 1e-9 multiplies G by 1 / R: its update fits no fixed-point unit
    (one carries 2^28).  R itself has an absolute rounding error of a few 2^-53, so G has a
    relative one of a few 2^-53 / R at best: 2^-53 64 / 1e-11 is the bound."""
    U, dtau = 8.0, 0.25
    bath, s, seed, at = near_singular_flip(L, U, dtau)
    cfg = dict(wl.CONFIGS["square6"], Lx=1, Ly=1, beta=L * dtau, dtau=dtau, U=U, chains_per_site=1,
               refresh_every=1000, bin_size=4, max_bins=1, seed=seed, n_matsubara=4)
    ctx = hf.Context(hf.make_params(cfg))
    for sp in range(2):
        hf.hf_set_g0(ctx.handle, 0, sp, bath[sp])
    hf.hf_set_fields(ctx.handle, s[None].astype(np.int8), np.zeros(1, dtype=np.uint32))
    hf.hf_sweep(ctx.handle, 0, 0, 1)
    G0 = hf.hf_get_green(ctx.handle, 0, L)
    hf.hf_sweep(ctx.handle, 1, 0, 0)
    hf.hf_sync(ctx.handle)
    s1 = hf.hf_get_fields(ctx.handle, 1, L)[0][0]
    G1 = hf.hf_get_green(ctx.handle, 0, L)
    ctx.close()
    assert s1[at] == -s[at] and np.array_equal(np.delete(s1, at), np.delete(s, at))
    _, lam = o.constants(L * dtau, U, L)
    u = np.array([o.uniform(seed, 0, 0, 0, l) for l in range(L)])
    e, e64, q = np.zeros((1, 2)), np.zeros((1, 2)), np.zeros((1, L), dtype=np.int8)
    dp = lambda x: x.ctypes.data_as(C.POINTER(C.c_double))
    i8 = lambda x: x.ctypes.data_as(C.POINTER(C.c_int8))
    s0 = np.ascontiguousarray(s[None], dtype=np.int8)
    helper.green_errors(L, 1, 1, C.c_double(np.exp(-2 * lam) - 1), C.c_double(np.exp(2 * lam) - 1), dp(G0),
                        i8(s0), dp(u), dp(G1), dp(e), dp(e64), i8(q))
    assert np.array_equal(q[0], s1)
    assert np.abs(G1[0]).max() > 1e8
    assert e.max() <= 64 * 2.0 ** -53 / 1e-11, (e, e64)
