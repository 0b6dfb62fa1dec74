"""Steps whose kernel is chosen by size, on both sides of each line, against
the generic kernel bit for bit (every FP32 kernel runs the same explicitly
rounded arithmetic)."""
import numpy as np
import pytest

from paper_2006_15932_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,ny,ns,bc", [
    (513, 113, 2, (W.PERIODIC, W.OUTFLOW)),  # 9 x 15 pair tiles, ragged both ways
    (512, 128, 2, (W.OUTFLOW, W.PERIODIC)),  # exactly 128 pair tiles
    (510, 119, 2, (W.OUTFLOW, W.OUTFLOW)),   # 120: two threads per pair
    (67, 9, 2, (W.PERIODIC, W.PERIODIC)), (33, 5, 2, (W.OUTFLOW, W.PERIODIC)), (1, 1, 2, (W.PERIODIC, W.OUTFLOW)),
    (31, 6, 4, (W.OUTFLOW, W.OUTFLOW)), (97, 75, 4, (W.PERIODIC, W.PERIODIC)),
    (1025, 65, 1, (W.PERIODIC, W.PERIODIC)),
    (321, 200, 3, (W.OUTFLOW, W.PERIODIC)),
    (130, 300, 4, (W.PERIODIC, W.OUTFLOW)),
])
def test_automatic_step_matches_generic_bitwise(orc, nx, ny, ns, bc):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2006_15932_gb300 import build as B
    from paper_2006_15932_gb300 import dbm as D

    B.build()
    pb = W.random_smooth(nx, ny, ns, seed=3, reactive=ns == 3, force=ns in (2, 4), bc=bc)
    p = orc.params_of(pb)
    f0 = orc.init_feq(p, pb.rho_s, pb.ux, pb.uy, pb.T)
    f0 = f0 * (1.0 + 0.05 * np.random.default_rng(4).uniform(-1, 1, f0.shape))
    out = {}
    for kern in ("generic", "auto"):
        s = D.Solver(pb, "fp32", step_kernel=kern)
        s.set_f(f0)
        s.step(5)
        out[kern] = s.get_f()
        assert s.status() == (0, 0)
        s.close()
    assert torch.equal(out["auto"], out["generic"])


@pytest.mark.parametrize("prec,ns", [("fp32", 1), ("fp32", 2), ("fp32", 5), ("fp64", 2), ("bf16dev", 2)])
def test_chained_steps_captured_and_beside_another_stream(prec, ns):
    """Steps launched with programmatic serialization: captured into a graph
    and replayed, and interleaved with a second solver on another stream, they
    give the bits of plain steps."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2006_15932_gb300 import build as B
    from paper_2006_15932_gb300 import dbm as D

    B.build()
    pb = W.random_smooth(131, 67, ns, seed=8)
    side = torch.cuda.Stream()
    plain, graphed, beside = (D.Solver(pb, prec, stream=st) for st in (None, None, side))
    for s in (plain, graphed, beside):
        s.set_state()
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):  # captured, not run: four steps from the first buffer
        graphed.step(4)
    graph.replay()
    graph.replay()
    for _ in range(4):
        beside.step(2)
        plain.step(2)
    torch.cuda.synchronize()
    want = plain.get_f()
    assert torch.equal(graphed.get_f(), want) and torch.equal(beside.get_f(), want)
    for s in (plain, graphed, beside):
        assert s.status() == (0, 0)
        s.close()
