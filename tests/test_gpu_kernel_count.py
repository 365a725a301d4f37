"""`sbp_linear_backward_kernel_count` against the kernels that the call puts into a captured graph."""
import pytest
import torch

import paper_2210_00129_b200 as sbp

pytestmark = pytest.mark.gpu


def _nodes(graph):
    from cuda.bindings import runtime
    raw = runtime.cudaGraph_t(graph.raw_cuda_graph())
    err, _, n = runtime.cudaGraphGetNodes(raw, 0)
    assert int(err) == 0
    err, nodes, n = runtime.cudaGraphGetNodes(raw, n)
    assert int(err) == 0
    kinds = [runtime.cudaGraphNodeGetType(node)[1] for node in nodes[:n]]
    assert all(k == runtime.cudaGraphNodeType.cudaGraphNodeTypeKernel for k in kinds)
    return n


FLAGS = [0, sbp.SBP_FLAG_ACCUMULATE, sbp.SBP_FLAG_W_OUT_IN, sbp.SBP_FLAG_W_OUT_IN | sbp.SBP_FLAG_ACCUMULATE, sbp.SBP_FLAG_PLAIN_FMA,
         sbp.SBP_FLAG_VALIDATE | sbp.SBP_FLAG_W_OUT_IN | sbp.SBP_FLAG_ACCUMULATE, sbp.SBP_FLAG_DY_COMPACT]


@pytest.mark.parametrize("code,M_keep,C_in,C_out", [
    (0, 30, 36, 68), (0, 3000, 64, 64), (0, 500, 768, 768), (1, 20, 64, 32), (1, 294, 264, 136), (1, 3000, 64, 512), (1, 392, 768, 768),
    (1, 6272, 768, 768), (1, 3000, 128, 256),
])
def test_count_is_what_the_call_launches(code, M_keep, C_in, C_out):
    M = 2 * M_keep
    tdt = torch.bfloat16 if code else torch.float32
    z = lambda *shape, dtype=tdt: torch.zeros(*shape, dtype=dtype, device="cuda")
    Xk, dY, W, dX = z(M_keep, C_in), z(M, C_out), z(C_in * C_out), z(M, C_in)
    dW, db, status = z(C_in * C_out, dtype=torch.float32), z(C_out, dtype=torch.float32), z(1, dtype=torch.int32)
    rows = torch.arange(M_keep, dtype=torch.int32, device="cuda") * 2
    nb = sbp.sbp_linear_backward_workspace_bytes(code, M, M_keep, C_in, C_out)
    ws = torch.empty(nb, dtype=torch.uint8, device="cuda")
    for flags in FLAGS:
        for want in ("wbx", "wx", "wb", "bx", "w", "b", "x"):
            def call():
                sbp.sbp_linear_backward(code, Xk, dY, W, rows, None, M, M_keep, C_in, C_out, dW if "w" in want else None,
                                        db if "b" in want else None, dX if "x" in want else None, flags, ws, nb, status)
            call()
            torch.cuda.synchronize()
            graph = torch.cuda.CUDAGraph(keep_graph=True)
            with torch.cuda.graph(graph):
                call()
            count = sbp.sbp_linear_backward_kernel_count(code, M, M_keep, C_in, C_out, "w" in want, "b" in want, "x" in want, flags)
            assert _nodes(graph) == count, (flags, want)
