"""A tile shape that a caller sets is the one that runs, in every precision that has shapes: the
threads per CTA of the captured launch are those that dk_gram_config_info reports. And the
built-in choice where shape 17 gives an SM one or two CTAs."""
import ctypes

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


class _KernelNode(ctypes.Structure):  # CUDA_KERNEL_NODE_PARAMS_v2
    _fields_ = [("func", ctypes.c_void_p), ("grid", ctypes.c_uint * 3), ("block", ctypes.c_uint * 3),
                ("smem", ctypes.c_uint), ("params", ctypes.c_void_p), ("extra", ctypes.c_void_p),
                ("kern", ctypes.c_void_p), ("ctx", ctypes.c_void_p)]


def _launched_threads(torch, call):
    """Threads per CTA of each kernel that `call` launches, from a capture of it."""
    cu = ctypes.CDLL("libcuda.so.1")
    call()  # lazy loading and workspaces before the capture
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph(keep_graph=True)
    with torch.cuda.graph(g):
        call()
    graph = ctypes.c_void_p(g.raw_cuda_graph())
    n = ctypes.c_size_t(0)
    assert cu.cuGraphGetNodes(graph, None, ctypes.byref(n)) == 0
    nodes = (ctypes.c_void_p * n.value)()
    assert cu.cuGraphGetNodes(graph, nodes, ctypes.byref(n)) == 0
    threads = []
    for node in nodes:
        kind, par = ctypes.c_int(-1), _KernelNode()
        assert cu.cuGraphNodeGetType(ctypes.c_void_p(node), ctypes.byref(kind)) == 0
        if kind.value == 0:  # CU_GRAPH_NODE_TYPE_KERNEL
            assert cu.cuGraphKernelNodeGetParams_v2(ctypes.c_void_p(node), ctypes.byref(par)) == 0
            threads.append(par.block[0])
    return threads


# 40 samples: few enough for the lanes form; 230: where the built-in choice is the small FP64 tiles
@pytest.mark.parametrize("m", [40, 230])
@pytest.mark.parametrize("c128,chi,cid", [(True, 4, 1), (False, 4, 1), (False, 4, 17), (False, 4, 22), (False, 8, 1)])
def test_set_shape_runs(c128, chi, cid, m):
    import torch
    from paper_2602_01330_gb300 import build, dualk, synthetic
    build.build()
    ctx = dualk.Context(0)
    dtype = dualk.DK_C128 if c128 else dualk.DK_C64
    x = torch.from_numpy(synthetic.uniform_angles(m, 6, seed=9, dtype=np.float32)).cuda()
    mps = dualk.mps_build(ctx, x, dualk.FeatureMap(reps=3 if chi == 8 else 2, chi_max=chi), dtype=dtype)
    ctx.set_gram_config(cid)
    _, _, threads = dualk.gram_config_info(cid, dtype, chi)
    got = _launched_threads(torch, lambda: dualk.gram(ctx, mps, refine=None))
    ctx.set_gram_config(0)
    assert got == [threads]
    ctx.sync_status()
    ctx.close()


# blocks of 16 x 16 tiles that give an SM one to two CTAs and for which the narrower shapes need more
# waves or more than a quarter of one: measured at n = 784, us, shape 17 against the best other:
# 634 / 667, 650 / 671, 650 / 689, 653 / 690, 651 / 687, 651 / 689
@pytest.mark.parametrize("rows,m", [(80, 500), (100, 500), (130, 500), (64, 1000), (0, 333), (0, 366)])
def test_built_in_choice_with_two_tiles_to_an_sm(rows, m):
    import torch
    from paper_2602_01330_gb300 import build, dualk, synthetic
    if torch.cuda.get_device_properties(0).multi_processor_count != 152:
        pytest.skip("sizes chosen for 152 SMs")
    build.build()
    ctx = dualk.Context(0)
    x = torch.from_numpy(synthetic.uniform_angles(m + rows, 6, seed=9, dtype=np.float32)).cuda()
    cols = dualk.mps_build(ctx, x[:m].contiguous(), dualk.FeatureMap())
    if rows:
        test = dualk.mps_build(ctx, x[m:].contiguous(), dualk.FeatureMap())
        got = _launched_threads(torch, lambda: dualk.dual_kernel_rows(ctx, test, cols, refine=None))
    else:
        got = _launched_threads(torch, lambda: dualk.gram(ctx, cols, refine=None))
    assert got == [dualk.gram_config_info(17)[2]] != [dualk.gram_config_info(19)[2]]
    ctx.sync_status()
    ctx.close()


@pytest.mark.parametrize("n,m,shape", [(4, 122, 2), (4, 100, None), (16, 122, None)])
def test_built_in_choice_bond8(n, m, shape):
    """122 samples are 49 pairs per SM: tiles below 12 qubits, lanes (128 threads) from there on."""
    import torch
    from paper_2602_01330_gb300 import build, dualk, synthetic
    if torch.cuda.get_device_properties(0).multi_processor_count != 152:
        pytest.skip("sizes chosen for 152 SMs")
    build.build()
    ctx = dualk.Context(0)
    x = torch.from_numpy(synthetic.uniform_angles(m, n, seed=9, dtype=np.float32)).cuda()
    mps = dualk.mps_build(ctx, x, dualk.FeatureMap(reps=3, chi_max=8))
    want = 128 if shape is None else dualk.gram_config_info(shape, dualk.DK_C64, 8)[2]
    assert _launched_threads(torch, lambda: dualk.gram(ctx, mps, refine=None)) == [want]
    ctx.sync_status()
    ctx.close()
