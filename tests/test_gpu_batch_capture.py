"""lbm_batch_step keeps its steps in host-side budgets and buffer indices, which
a replayed CUDA graph would not move: it refuses a stream that is being
captured, however many domains step, and steps as usual afterwards."""
import numpy as np
import pytest

from paper_1705_10045_gb300 import lbm
from paper_1705_10045_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("lattice,shape", [(9, (1, 40, 40)), (19, (20, 20, 20))])
@pytest.mark.parametrize("domains", [1, 2])
def test_a_captured_stream_is_refused(lattice, shape, domains):
    import torch
    f = W.spinodal(shape, rho0=0.9, T0=0.8, noise=2e-2, seed=5)
    u = np.ascontiguousarray(f.u[: 2 if lattice == 9 else 3])
    kw = dict(nx=shape[2], ny=shape[1], nz=shape[0])
    stream = torch.cuda.Stream()
    batch = lbm.LbmBatch(lattice=lattice, storage=lbm.LBM_STORE_FP32, stream=stream.cuda_stream)
    sim = lbm.Lbm(lattice=lattice, storage=lbm.LBM_STORE_FP32, **kw)
    buf = torch.zeros(1000, device="cuda")
    try:
        ids = [batch.add(f.rho, u, 1.5 * f.T, 9, **kw) for _ in range(domains)]
        batch.step(3)
        batch.sync()
        torch.cuda.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=stream, capture_error_mode="relaxed"):
            buf.add_(1)
            with pytest.raises(lbm.LbmError, match="captured"):
                batch.step(3)
        graph.replay()
        torch.cuda.synchronize()
        assert float(buf.sum()) == 1000
        for i in ids:
            assert batch.status(i) == (3, 6)
        batch.step(6)
        sim.init(f.rho, u, 1.5 * f.T)
        sim.step(9)
        for i in ids:
            assert batch.status(i) == (9, 0)
            assert np.array_equal(sim.get_state(), batch.get_state(i))
    finally:
        batch.close()
        sim.close()
