"""Conserved totals of float states keep what FP64 additions of the values keep.

1. Values that are multiples of 2^-50 with magnitudes adding up to less than 8:
   FP64 adds them in any order without rounding, so a total formed in at least
   53 bits is the exact sum, bit for bit.
2. Signed values over ten decades: the kernel adds a thread's cells exactly up
   to 2^-60 of their magnitudes and behind that makes at most 7 FP64 additions
   per group of 16 cells (one group per thread here), 5 of the warp, 8 of the
   block, 12 over the rings and 16 S + 4 of the final kernel, each 2^-53 of the
   magnitudes added: fewer than 64 of them, 2^-47.
3. Magnitudes whose sum leaves the float range: finite, and within 2^-47 too.
"""
import numpy as np
import pytest

from paper_2006_15932_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _solver(nx, ny, ns=1):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2006_15932_gb300 import build as B
    from paper_2006_15932_gb300 import dbm as D

    B.build()
    pb = W.random_smooth(nx, ny, ns, seed=2)
    for sp in pb.species:
        sp.m = 1.0
    return pb, D.Solver(pb, "fp32")


def _wide(rng, n):
    """n x 16 floats, multiples of 2^-50, of magnitude 2^-27 to 2^-1 or so."""
    k = rng.integers(2**23, 2**24, (n, 16)) * rng.choice([-1.0, 1.0], (n, 16))
    return k * 2.0 ** rng.choice([-27, -35, -43, -50], (n, 16))


@pytest.mark.parametrize("nx,ny", [(4, 1), (7, 1), (1, 5)])
def test_mass_is_exact_where_fp64_additions_are(nx, ny):
    rng = np.random.default_rng(nx)
    pb, s = _solver(nx, ny)
    for _ in range(32):
        f = np.zeros((1, 16, ny, nx))
        for c, v in zip(rng.permutation(nx * ny)[:4], _wide(rng, 4)):
            f[0, :, c // nx, c % nx] = v
        assert np.abs(f).sum() < 8.0
        s.set_f(f)
        assert float(s.conservation()[0]) == float(f.sum())
    s.close()


def test_mass_is_exact_across_a_threads_groups():
    """2200^2 cells: 1 210 000 vectors of four cells on 512 x 256 threads, so a
    thread takes up to ten vectors, past the eight of one group."""
    nx = ny = 2200
    pb, s = _solver(nx, ny)
    rng = np.random.default_rng(1)
    nv = nx // 4
    f = np.zeros((1, 16, ny * nx))
    for first in (0, 5, 37_000, 38_211):  # the thread's first vector
        vec = first + 131_072 * np.arange(10)
        vec = vec[vec < nv * ny]
        cells = (vec // nv) * nx + 4 * (vec % nv) + rng.integers(0, 4, len(vec))
        f[:] = 0.0
        f[0][:, cells] = _wide(rng, len(vec)).T
        assert np.abs(f[0][:, cells]).sum() < 8.0
        s.set_f(f.reshape(1, 16, ny, nx))
        assert float(s.conservation()[0]) == float(f[0][:, cells].sum())
    s.close()


@pytest.mark.parametrize("top", [1.0, 1.0e38])
def test_totals_of_mixed_magnitudes(top):
    """top = 1e38: a cell's ring, and a velocity over a thread's cells, add up
    to more than the largest float."""
    nx, ny, ns = 33, 9, 2
    pb, s = _solver(nx, ny, ns)
    rng = np.random.default_rng(3)
    f = rng.uniform(0.5, 1.0, (ns, 16, ny, nx)) * rng.choice([-1.0, 1.0], (ns, 16, ny, nx))
    f *= 10.0 ** -rng.uniform(0.0, 10.0, f.shape)
    if top > 1.0:
        f = np.ones_like(f)
    f = (f * top).astype(np.float32).astype(np.float64)
    s.set_f(f)
    got = s.conservation().cpu().numpy()
    dirs = [((1, 0), (0, 1), (-1, 0), (0, -1)), ((1, 1), (-1, 1), (-1, -1), (1, -1))]
    want, size = np.zeros(ns + 3, np.longdouble), np.zeros(ns + 3, np.longdouble)
    for q, sp in enumerate(pb.species):
        for i in range(16):
            (dx, dy), v = dirs[(i // 4) % 2][i % 4], sp.v[i // 4]
            e = 0.5 * ((dx * dx + dy * dy) * v * v + sp.eta[i // 4] ** 2)
            total, mag = f[q, i].astype(np.longdouble).sum(), np.abs(f[q, i]).astype(np.longdouble).sum()
            for k, w in ((q, 1.0), (ns, dx * v), (ns + 1, dy * v), (ns + 2, e)):
                want[k] += w * total
                size[k] += abs(w) * mag
    assert np.all(np.isfinite(got))
    assert np.all(np.abs(got[: ns + 3] - want) <= 2.0**-47 * size), (got[: ns + 3] - want) / size
    s.close()
