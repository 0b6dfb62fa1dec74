"""The bounded wait of the two-thread step, and the bounds-checked build on the
kernels that the automatic choice runs on small and on larger grids of two and
four species.

The timeout: a handle made with wait_polls < 0 polls its first tile copy zero
times, so every CTA reports at once, waits (bounded) for its valid copies and
leaves without writing.  Nothing faults or hangs.
"""
import json
import os
import subprocess
import sys

import numpy as np
import pytest

from paper_2006_15932_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CASES = [  # name, nx, ny, species, kernel, the kernel that runs
    ("half_s2_37x13", 37, 13, 2, "auto", "k_step_half<2,32,4>"),
    ("half_s2_101x50", 101, 50, 2, "auto", "k_step_half<2,32,4>"),
    ("half_s4_37x13", 37, 13, 4, "auto", "k_step_half<4,32,4>"),
    ("cell_s4_37x13", 37, 13, 4, "tma_cell", "k_step_tma<4,32,7,1>"),
    ("cell_s4_130x9", 130, 9, 4, "tma_cell", "k_step_tma<4,32,7,1>"),
    ("pair_s2_513x113", 513, 113, 2, "auto", "k_step_tma<2,64,8,2>"),
    ("staged_pair_s5_67x9", 67, 9, 5, "tma_pair", "k_step_staged<5,64,8,2>"),
]


def _dbm():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2006_15932_gb300 import build as B
    from paper_2006_15932_gb300 import dbm as D

    B.build()
    return D


@pytest.mark.parametrize("ns", [2, 4])
def test_two_thread_step_reports_its_timeout(orc, ns):
    D = _dbm()
    pb = W.random_smooth(70, 20, ns, seed=5, force=ns == 4)
    s = D.Solver(pb, "fp32", wait_polls=-1)
    assert s.step_kernel_name() == f"k_step_half<{ns},32,4>"
    s.set_state()
    f0 = s.get_f()
    s.step(2)  # each step leaves its output buffer as it was; the first buffer is current again
    rc, bits = s.status()
    assert rc == -8 and bits & 16, (rc, bits)
    assert torch.equal(s.get_f(), f0)
    s.close()
    ok = D.Solver(pb, "fp32")
    ok.set_state()
    ok.step(3)
    assert ok.status() == (0, 0)
    p = orc.params_of(pb)
    ref, st = orc.run(p, orc.init_feq(p, pb.rho_s, pb.ux, pb.uy, pb.T), 3)
    f = ok.get_f().cpu().numpy()
    assert st == 0 and np.max(np.abs(f - ref)) / np.max(np.abs(ref)) <= 2e-5
    ok.close()


def run_cases(out_dir):
    from paper_2006_15932_gb300 import dbm as D

    D.load()
    bits = {}
    for name, nx, ny, ns, kern, runs in CASES:
        for k, bc in enumerate(((W.PERIODIC, W.OUTFLOW), (W.OUTFLOW, W.PERIODIC))):
            s = D.Solver(W.random_smooth(nx, ny, ns, seed=nx + ny, force=ns == 4, bc=bc), "fp32", step_kernel=kern)
            assert s.step_kernel_name() == runs
            s.set_state()
            s.step(4)
            bits[f"{name}_{k}"] = s.status()[1]
            np.save(os.path.join(out_dir, f"{name}_{k}.npy"), s.get_f().cpu().numpy())
            s.close()
    return bits


def test_checked_build_finds_no_out_of_range_index(tmp_path):
    _dbm()
    from paper_2006_15932_gb300 import build as B

    lib = B.build(checked=True)
    checked, plain = tmp_path / "checked", tmp_path / "plain"
    checked.mkdir()
    plain.mkdir()
    code = ("import json, sys; sys.path.insert(0, %r); "
            "from tests.test_gpu_wait_paths import run_cases; print(json.dumps(run_cases(%r)))") % (ROOT, str(checked))
    r = subprocess.run([sys.executable, "-c", code], env=dict(os.environ, DBM_LIB=lib), capture_output=True, text=True,
                       timeout=600)
    assert r.returncode == 0, r.stderr[-3000:]
    bits = json.loads(r.stdout.strip().splitlines()[-1])
    assert all(b == 0 for b in bits.values()), bits
    bits = run_cases(str(plain))
    assert all(b == 0 for b in bits.values()), bits
    for name in bits:
        assert np.array_equal(np.load(plain / (name + ".npy")), np.load(checked / (name + ".npy"))), name
