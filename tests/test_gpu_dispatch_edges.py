"""The size lines that follow the device's SM count, from both sides: the kernel
that runs, and its result (FP32 against the generic kernel bit for bit, FP64
against the oracle at the tolerance of tests/test_gpu_f64.py)."""
import numpy as np
import pytest

from paper_2006_15932_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _setup():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2006_15932_gb300 import build as B
    from paper_2006_15932_gb300 import dbm as D

    B.build()
    return D, torch.cuda.get_device_properties(0).multi_processor_count


@pytest.mark.parametrize("ns,wide,over", [(2, 3, 0), (2, 3, 1), (4, 1, 0), (4, 1, 1)])
def test_two_thread_step_up_to_its_share_of_the_chip(orc, ns, wide, over):
    """`wide` columns of 32 x 4 tiles, one row of them per SM (and one more)."""
    D, sms = _setup()
    nx, ny = 32 * wide - 1, 4 * sms - 1 + 4 * over
    want = f"k_step_half<{ns},32,4>" if not over else "k_step_tma<2,64,8,2>" if ns == 2 else "k_step_tma<4,32,7,1>"
    pb = W.random_smooth(nx, ny, ns, seed=6, bc=(W.OUTFLOW, W.PERIODIC))
    f0 = orc.init_feq(orc.params_of(pb), pb.rho_s, pb.ux, pb.uy, pb.T)
    out = {}
    for kern in ("generic", "auto"):
        s = D.Solver(pb, "fp32", step_kernel=kern)
        if kern == "auto":
            assert s.step_kernel_name() == want
        s.set_f(f0)
        s.step(4)
        assert s.status() == (0, 0)
        out[kern] = s.get_f()
        s.close()
    assert torch.equal(out["auto"], out["generic"])


@pytest.mark.parametrize("over", [0, 1])
def test_fp64_small_grid_step_up_to_four_ctas_per_sm(orc, over):
    D, sms = _setup()
    pb = W.random_smooth(16 * sms + over, 1, 2, seed=8, bc=(W.PERIODIC, W.PERIODIC))
    p = orc.params_of(pb)
    f0 = orc.init_feq(p, pb.rho_s, pb.ux, pb.uy, pb.T)
    s = D.Solver(pb, "fp64")
    assert s.step_kernel_name() == ("k_step_f64<2>" if over else "k_step_f64_small<2>")
    s.set_f(f0)
    s.step(3)
    got = s.get_f().cpu().numpy()
    want, st = orc.run(p, f0, 3)
    assert st == 0 and s.status() == (0, 0)
    assert np.max(np.abs(got - want)) <= 1e-14 * np.max(np.abs(want))
    s.close()
