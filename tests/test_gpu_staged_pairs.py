"""Five and more species with two cells per thread when asked for: the kernel
that runs, and its bits against the generic kernel (ragged tiles, odd nx, one
and several 64 x 8 tiles)."""
import numpy as np
import pytest

from paper_2006_15932_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("ns,nx,ny,force,bc", [(5, 67, 9, True, (W.PERIODIC, W.PERIODIC)),
                                               (6, 33, 11, False, (W.OUTFLOW, W.PERIODIC)),
                                               (7, 1, 3, True, (W.OUTFLOW, W.OUTFLOW)),
                                               (8, 130, 17, False, (W.PERIODIC, W.OUTFLOW))])
def test_tma_pair_steps_two_cells_per_thread(orc, ns, nx, ny, force, bc):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2006_15932_gb300 import build as B
    from paper_2006_15932_gb300 import dbm as D

    B.build()
    pb = W.random_smooth(nx, ny, ns, seed=3, force=force, bc=bc)
    f0 = orc.init_feq(orc.params_of(pb), pb.rho_s, pb.ux, pb.uy, pb.T)
    f0 = f0 * (1.0 + 0.05 * np.random.default_rng(4).uniform(-1, 1, f0.shape))
    out = {}
    for kern in ("generic", "tma_pair"):
        s = D.Solver(pb, "fp32", step_kernel=kern)
        if kern == "tma_pair":
            assert s.step_kernel_name() == f"k_step_staged<{ns},64,8,2>"
        s.set_f(f0)
        s.step(5)
        assert s.status() == (0, 0)
        out[kern] = s.get_f()
        s.close()
    assert torch.equal(out["tma_pair"], out["generic"])
