"""Host threads that plan and launch the same kernel for graphs of different size at the same time (handles are
shared by threads; each thread here has a workspace of its own)."""
import ctypes
import threading

import pytest

from paper_2011_12453_gb300 import build as B, gna, workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch():
    import torch as t

    B.build()
    t.cuda.set_device(0)
    return t


@pytest.mark.parametrize("prec,op", [(gna.PREC_BF16X2, gna.OP_FORWARD), (gna.PREC_BF16X2, gna.OP_ELOC_INCR),
                                     (gna.PREC_BF16X2, gna.OP_METROPOLIS), (gna.PREC_BF16X2, gna.OP_BACKWARD),
                                     (gna.PREC_BF16, gna.OP_ELOC_INCR), (gna.PREC_FP32, gna.OP_ELOC_INCR),
                                     (gna.PREC_FP32, gna.OP_METROPOLIS), (gna.PREC_FP32, gna.OP_BACKWARD),
                                     (gna.PREC_FP64, gna.OP_ELOC_INCR), (gna.PREC_FP64, gna.OP_METROPOLIS)])
def test_two_sizes_at_once(torch, prec, op):
    model = gna.Model(16, 2, prec)
    theta = torch.tensor(W.random_theta(16, 2, seed=1), dtype=model.theta_dtype(), device="cuda")
    L, status = gna.lib(), []

    def work(g, calls, queries):
        torch.cuda.set_device(0)
        graph = gna.Graph.from_workload(g, 2)
        s = torch.tensor(W.random_spins(g.n_sites, 2, seed=4), device="cuda")
        out = torch.zeros(max(4, model.num_params), dtype=torch.float64, device="cuda")
        cot = torch.ones((2, 2), dtype=torch.float64, device="cuda")
        ws = torch.empty(max(256, gna.workspace_size(graph, model, op, 2)), dtype=torch.uint8, device="cuda")
        st = torch.cuda.Stream()
        torch.cuda.synchronize()
        head = (graph.handle, ctypes.byref(model.desc), theta.data_ptr(), s.data_ptr(), 2)
        tail = (ws.data_ptr(), ws.numel(), st.cuda_stream)
        call = {gna.OP_FORWARD: lambda: L.gna_forward(*head, out.data_ptr(), *tail),
                gna.OP_ELOC_INCR: lambda: L.gna_local_energy(*head, gna.ELOC_INCREMENTAL, out.data_ptr(), None, *tail),
                gna.OP_METROPOLIS: lambda: L.gna_metropolis_sweep(*head, 1, 0, 7, 0, None, 0.0, None, None, None, None, *tail),
                gna.OP_BACKWARD: lambda: L.gna_backward(*head, cot.data_ptr(), out.data_ptr(), *tail)}[op]
        n = ctypes.c_size_t(0)
        for _ in range(calls):
            status.append(call())
            for _ in range(queries):
                L.gna_workspace_size(graph.handle, ctypes.byref(model.desc), op, 2, ctypes.byref(n))
        st.synchronize()

    threads = [threading.Thread(target=work, args=a) for a in ((W.kagome(6), 1500, 0), (W.two_site(), 1500, 3))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert len(status) == 3000 and set(status) == {gna.GNA_OK}
