"""dbm_step_kernel_name against the kernel a step really enqueues: the step is
captured into a CUDA graph (not run) and the graph's kernel node names its
function."""
import re

import pytest

from paper_2006_15932_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _enqueued(solver, path):
    """The step kernel of one captured step, as 'name<a,b,...>' (integer
    template arguments)."""
    graph = torch.cuda.CUDAGraph(keep_graph=True)
    graph.enable_debug_mode()
    with torch.cuda.graph(graph):
        solver.step(1)
    graph.debug_dump(str(path))
    found = set()
    for name, args in re.findall(r"(k_step\w*?)I((?:Li\d+E)+)", path.read_text()):  # mangled
        found.add(name + "<" + ",".join(re.findall(r"\d+", args)) + ">")
    for name, args in re.findall(r"(k_step\w*)<(\d+(?:, ?\d+)*)", path.read_text()):  # or demangled
        found.add(name + "<" + args.replace(" ", "") + ">")
    assert len(found) == 1, found
    return found.pop()


@pytest.mark.filterwarnings("ignore:DEBUG")
@pytest.mark.parametrize("prec,nx,ny,ns,kern,opts", [
    ("fp32", 70, 20, 1, "auto", {}),
    ("fp32", 70, 20, 2, "auto", {}), ("fp32", 510, 119, 2, "auto", {}),
    ("fp32", 512, 128, 2, "auto", {}), ("fp32", 70, 20, 2, "tma_cell", {}), ("fp32", 70, 20, 2, "tma_pair", {}),
    ("fp32", 70, 20, 2, "tma_staged", {}), ("fp32", 70, 20, 2, "generic", {}),
    ("fp32", 512, 128, 2, "auto", {"rounding": "stochastic"}),
    ("fp32", 70, 20, 3, "auto", {}), ("fp32", 70, 20, 3, "tma_pair", {}),
    ("fp32", 70, 20, 4, "auto", {}), ("fp32", 400, 200, 4, "auto", {}), ("fp32", 70, 20, 4, "tma_cell", {}),
    ("fp32", 70, 20, 5, "auto", {}), ("fp32", 70, 20, 8, "tma", {}), ("fp32", 70, 20, 6, "tma_staged", {}),
    ("fp32", 70, 20, 5, "tma_pair", {}), ("fp32", 70, 20, 6, "generic", {}),
    ("fp64", 70, 20, 2, "auto", {}), ("fp64", 170, 20, 2, "auto", {}),
    ("bf16dev", 70, 20, 2, "auto", {}),
])
def test_reported_step_kernel_is_the_one_enqueued(tmp_path, prec, nx, ny, ns, kern, opts):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2006_15932_gb300 import build as B
    from paper_2006_15932_gb300 import dbm as D

    B.build()
    s = D.Solver(W.random_smooth(nx, ny, ns, seed=4), prec, step_kernel=kern, **opts)
    s.set_state()
    s.step(1)  # kernel attributes and modules outside the capture
    torch.cuda.synchronize()
    assert s.step_kernel_name() == _enqueued(s, tmp_path / "step.dot")
    s.close()
