"""The output calls at the edges of their kernels: conversion of stored
floats by bits, the ring-sum conservation totals on ragged vectors of four
cells, and the nonequilibrium moments of one to eight species.

Tolerances.  get_f is exact.  Conserved totals: every addition of the float
path is an exact float-float pair up to 2^-47 of its running sum and the FP64
additions behind it (at most 64 per thread, then 5 + 8 + 21 levels of tree)
add 2^-53 each of the running sum, so the total is within 2^-44 of the sum of
the magnitudes added.  Nonequilibrium moments of an FP64 state: the oracle's
own bound, 1e-12 of the largest moment of the same order (the difference
M f - f-hat cancels).
"""
import numpy as np
import pytest

from paper_2006_15932_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def D():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2006_15932_gb300 import build as B
    from paper_2006_15932_gb300 import dbm

    B.build()
    dbm.load()
    return dbm


def _state(orc, pb, seed=3):
    p = orc.params_of(pb)
    f = orc.init_feq(p, pb.rho_s, pb.ux, pb.uy, pb.T)
    return p, f * (1.0 + 0.05 * np.random.default_rng(seed).uniform(-1, 1, f.shape))


def test_stored_floats_are_read_back_exactly(D):
    pb = W.random_smooth(37, 5, 1)
    special = np.array([0.0, -0.0, 1.0, -1.0, 1e-38, 1.2e-38, 1e-40, -1e-45, 3.0e38, -3.0e38, np.inf, -np.inf],
                       dtype=np.float32)
    f = np.random.default_rng(1).choice(special, size=(1, 16, 5, 37)).astype(np.float64)
    s = D.Solver(pb, "fp32")
    s.set_f(f)
    got = s.get_f().cpu().numpy()
    assert np.array_equal(got, f) and np.array_equal(np.signbit(got), np.signbit(f))
    s.close()


@pytest.mark.parametrize("prec,nx,ny,ns", [("fp32", 1, 1, 1), ("fp32", 5, 3, 2), ("fp32", 1027, 515, 2),
                                           ("fp32", 34, 70, 3), ("fp32", 6, 9, 8), ("fp64", 1, 7, 2),
                                           ("fp64", 131, 66, 4), ("bf16dev", 67, 33, 2), ("bf16dev", 3, 2, 4)])
def test_conserved_totals(D, orc, prec, nx, ny, ns):
    pb = W.random_smooth(nx, ny, ns, seed=7, reactive=ns == 3)
    _, f = _state(orc, pb)
    s = D.Solver(pb, prec)
    s.set_f(f)
    f = s.get_f().cpu().numpy().astype(np.longdouble)
    want, size = np.zeros(ns + 4, np.longdouble), np.zeros(ns + 4, np.longdouble)
    dirs = [((1, 0), (0, 1), (-1, 0), (0, -1)), ((1, 1), (-1, 1), (-1, -1), (1, -1))]
    for q, sp in enumerate(pb.species):
        for i in range(16):
            r = i // 4
            dx, dy = dirs[r % 2][i % 4]
            v, total = sp.v[r], f[q, i].sum()
            e = 0.5 * ((dx * dx + dy * dy) * v * v + sp.eta[r] ** 2)
            for k, w in ((q, 1.0), (ns, dx * v), (ns + 1, dy * v), (ns + 2, e)):
                want[k] += sp.m * w * total
                size[k] += sp.m * abs(w) * np.abs(f[q, i]).sum()
            if pb.k_ov and q == pb.fuel:
                want[ns + 3] += pb.Q / abs(sp.a) * total
                size[ns + 3] += pb.Q / abs(sp.a) * np.abs(f[q, i]).sum()
    got = s.conservation().cpu().numpy()
    assert np.all(np.abs(got - want) <= 2.0**-44 * size), (got - want) / size
    s.close()


@pytest.mark.parametrize("ns", [1, 2, 3, 5, 8])
def test_nonequilibrium_of_every_species_count(D, orc, ns):
    pb = W.random_smooth(35, 11, ns, seed=9)
    p, f = _state(orc, pb)
    s = D.Solver(pb, "fp64")
    s.set_f(f)
    got = s.nonequilibrium().cpu().numpy()
    want = np.asarray(orc.nonequilibrium(p, f)).reshape(got.shape)
    scale = np.abs(want).max(axis=(1, 2)).reshape(ns, 20)
    scale = np.maximum(scale, np.abs(want).max(axis=(1, 2)).reshape(ns, 20)[:, 12:].max(axis=1, keepdims=True))
    assert np.all(np.abs(got - want) <= 1e-12 * scale.reshape(-1, 1, 1))
    s.close()
