"""Which kernels are launched cooperatively: those whose blocks wait across clusters, and no others (a cooperative launch cannot start behind its
predecessor's last blocks, and the profiler shows no time for one in clusters)."""
import pytest
import torch

from paper_2509_23436_b200 import binding as lot
from paper_2509_23436_b200 import synth

pytestmark = pytest.mark.gpu


def launches(call):
    """(cooperative, blocks of a cluster, blocks) of every kernel that `call` launches, from a captured graph."""
    rt, drv = pytest.importorskip("cuda.bindings.runtime"), pytest.importorskip("cuda.bindings.driver")
    graph = torch.cuda.CUDAGraph(keep_graph=True)
    with torch.cuda.graph(graph):
        call()
    raw = rt.cudaGraph_t(graph.raw_cuda_graph())
    err, _, count = rt.cudaGraphGetNodes(raw, 0)
    err, nodes, count = rt.cudaGraphGetNodes(raw, count)
    assert int(err) == 0
    found = []
    for node in nodes[:count]:
        if rt.cudaGraphNodeGetType(node)[1] != rt.cudaGraphNodeType.cudaGraphNodeTypeKernel:
            continue
        ids = rt.cudaLaunchAttributeID
        attr = [rt.cudaGraphKernelNodeGetAttribute(node, i)[1] for i in (ids.cudaLaunchAttributeCooperative, ids.cudaLaunchAttributeClusterDimension)]
        params = drv.cuGraphKernelNodeGetParams(drv.CUgraphNode(int(node)))[1]        # the runtime's form knows only its own copy's kernels
        found.append((bool(attr[0].cooperative), max(1, attr[1].clusterDim.x), params.gridDimX * params.gridDimY * params.gridDimZ))
    return found


# B, H, n, d, r, dtype, path, one cluster or none a problem
@pytest.mark.parametrize("B,H,n,d,r,dtype,path,one", [
    (1, 2, 1024, 64, 64, torch.bfloat16, 4, True), (1, 16, 4096, 64, 64, torch.bfloat16, 4, True), (1, 1, 30000, 64, 64, torch.bfloat16, 4, False),
    (1, 16, 1000, 64, 32, torch.float32, 0, True), (1, 8, 900, 32, 128, torch.bfloat16, 0, True), (1, 1, 30001, 16, 64, torch.float32, 0, False)])
def test_only_groups_of_several_clusters_are_cooperative(B, H, n, d, r, dtype, path, one):
    x = synth.make(B, H, n, d, r, seed=1, dtype=dtype, eps=0.1, iters=3)
    dev = torch.device("cuda:0")
    t = [getattr(x, name).to(dev) for name in ("q", "k", "v", "z", "beta")]
    assert lot.lot_path(lot.LOT_BF16 if dtype == torch.bfloat16 else lot.LOT_F32, B, H, n, d, r, 3) == path
    out, ws = lot.lot_attention_fwd_ex(*t, None, x.eps, x.iters)
    torch.cuda.synchronize()
    found = launches(lambda: lot.lot_attention_fwd_ex(*t, None, x.eps, x.iters, out=out, ws=ws))
    assert any(k > 1 for _, k, _ in found) or not one
    assert any(coop for coop, _, _ in found) == (not one)
