"""launches_per_step, kernel_launches and us_linear_group_launches against the kernel nodes of a captured step."""
import pytest
import torch

pytestmark = pytest.mark.gpu


def _kernels(fn):
    from cuda.bindings import driver as cu
    fn()
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph(keep_graph=True)
    with torch.cuda.graph(g):
        fn()
    graph = cu.CUgraph(g.raw_cuda_graph())
    err, _, n = cu.cuGraphGetNodes(graph, 0)
    err, nodes, n = cu.cuGraphGetNodes(graph, n)
    assert err == cu.CUresult.CUDA_SUCCESS
    return sum(cu.cuGraphNodeGetType(node)[1] == cu.CUgraphNodeType.CU_GRAPH_NODE_TYPE_KERNEL for node in nodes[:n])


@pytest.mark.parametrize("T,d,f,operand", [(256, 128, 512, "fp8"), (16000, 128, 400, "fp8"), (9000, 256, 768, "bf16"), (1000, 528, 2096, "fp8")])
def test_launches_of_an_ffn_step(T, d, f, operand):
    from paper_2303_11257_b200 import ffn
    blk = ffn.UnitScaledFFN(T, d, f, operand=operand)
    X, W1, W2, G = (torch.zeros(s, device="cuda") for s in ((T, d), (d, f), (f, d), (T, d)))
    assert _kernels(lambda: blk.step(X, W1, W2, G)) == blk.launches_per_step
    assert blk.launches_per_step == (4 if T >= 9000 else 3)             # the weight gradients' contractions in a launch of their own


@pytest.mark.parametrize("nseq,slen,nhead,attention,norm,fused", [(8, 256, 2, "bf16", None, False), (32, 256, 2, "fp8", "post", True), (40, 256, 2, "bf16", None, True)])
def test_launches_of_an_encoder_step(nseq, slen, nhead, attention, norm, fused):
    from paper_2303_11257_b200 import encoder
    T, d, f = nseq * slen, 64 * nhead, 256 * nhead
    layer = encoder.UnitScaledEncoderLayer(nseq, slen, d, nhead, f, attention=attention, fused_attention=fused, norm=norm)
    t = [torch.zeros(s, device="cuda") for s in ((T, d), (d, 3 * d), (d, d), (d, f), (f, d), (T, d))]
    ln = [torch.zeros(d, device="cuda") for _ in range(4)] if norm else None
    assert _kernels(lambda: layer.step(*t, ln=ln)) == layer.kernel_launches
