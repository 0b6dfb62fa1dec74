"""The FP64 step's two kernels (4 cells per CTA on small grids, 32 on the
rest) at their edges against the FP64 oracle.

Tolerance: the kernel evaluates every formula in the oracle's order, each
operation rounded as there, so one step differs only through the compilers'
exp (one ulp of the rate) and the oracle's own summation of M^-1's vanishing
entries: 1e-14 of the largest value after three steps.
"""
import numpy as np
import pytest

from paper_2006_15932_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,ny,ns,react,force,bc", [
    (1, 1, 1, False, True, (W.PERIODIC, W.OUTFLOW)), (7, 1, 2, False, False, (W.OUTFLOW, W.PERIODIC)),
    (2432, 1, 2, False, True, (W.PERIODIC, W.PERIODIC)), (2433, 1, 2, False, True, (W.PERIODIC, W.PERIODIC)),
    (33, 73, 3, True, True, (W.OUTFLOW, W.OUTFLOW)), (61, 41, 3, True, False, (W.PERIODIC, W.OUTFLOW)),
    (9, 5, 8, True, True, (W.OUTFLOW, W.PERIODIC)), (50, 50, 8, True, True, (W.PERIODIC, W.PERIODIC)),
    (3, 900, 5, False, True, (W.OUTFLOW, W.OUTFLOW)),
])
def test_fp64_splits_against_oracle(orc, nx, ny, ns, react, force, bc):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2006_15932_gb300 import build as B
    from paper_2006_15932_gb300 import dbm as D

    B.build()
    pb = W.random_smooth(nx, ny, ns, seed=31 + nx, reactive=react, force=force, bc=bc)
    p = orc.params_of(pb)
    f0 = orc.init_feq(p, pb.rho_s, pb.ux, pb.uy, pb.T)
    f0 = f0 * (1.0 + 0.05 * np.random.default_rng(2).uniform(-1, 1, f0.shape))
    s = D.Solver(pb, "fp64")
    s.set_f(f0)
    s.step(3)
    got = s.get_f().cpu().numpy()
    assert s.status() == (0, 0)
    want, st = orc.run(p, f0, 3)
    assert st == 0
    assert np.max(np.abs(got - want)) <= 1e-14 * np.max(np.abs(want))
    s.close()


def test_fp64_tiny_and_huge_values_keep_their_quotients(orc):
    """Densities near the ends of the range that the reciprocal path covers
    and beyond it: the step follows the oracle there too."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2006_15932_gb300 import dbm as D

    for scale in (1e-300, 1e-250, 1e-200, 1e200, 1e230):
        pb = W.random_smooth(37, 6, 2, seed=5)
        p = orc.params_of(pb)
        f0 = orc.init_feq(p, pb.rho_s, pb.ux, pb.uy, pb.T) * scale
        s = D.Solver(pb, "fp64")
        s.set_f(f0)
        s.step(2)
        got = s.get_f().cpu().numpy()
        want, st = orc.run(p, f0, 2)
        assert np.max(np.abs(got - want)) <= 1e-14 * np.max(np.abs(want)), scale
        s.close()
