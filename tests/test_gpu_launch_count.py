"""afqmc_kp_launch_count against the kernel nodes of the same call captured into a CUDA graph."""
import ctypes

import pytest

import gen

torch = pytest.importorskip("torch")
from gpu_util import dev, make  # noqa: E402

pytestmark = pytest.mark.gpu


def kernel_nodes(call):
    """Kernel nodes of the graph that `call` captures."""
    cu = ctypes.CDLL("libcuda.so.1")
    call()                       # one-time attributes outside the capture
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph(keep_graph=True)
    with torch.cuda.graph(g):
        call()
    graph, n = ctypes.c_void_p(g.raw_cuda_graph()), ctypes.c_size_t(0)
    assert cu.cuGraphGetNodes(graph, None, ctypes.byref(n)) == 0
    nodes = (ctypes.c_void_p * n.value)()
    assert cu.cuGraphGetNodes(graph, nodes, ctypes.byref(n)) == 0
    kernels = 0
    for node in nodes:
        kind = ctypes.c_int(-1)
        assert cu.cuGraphNodeGetType(ctypes.c_void_p(node), ctypes.byref(kind)) == 0
        kernels += kind.value == 0   # CU_GRAPH_NODE_TYPE_KERNEL
    return kernels


@pytest.mark.parametrize("nw", [1, 3])   # one walker: dE/dh in one chunk, without the sum over chunks
@pytest.mark.parametrize("precision", ["mixed", "fp64"])
def test_launch_count(precision, nw):
    sp = gen.SystemSpec(grid=(2, 1, 1), M=5, nocc=2, nchol=4, nwalkers=nw, random_trial=True, seed=3)
    sys_, _ = make(sp, precision)
    phi, g = dev(gen.near_trial_walkers(sp)), dev(gen.upstream(sp))
    x, w = dev(gen.fields(sp, 0)), torch.ones(nw, dtype=torch.float64, device="cuda")
    eloc = torch.empty((nw, 3), dtype=torch.complex128, device="cuda")
    ld = torch.empty((nw, 2), dtype=torch.complex128, device="cuda")
    gphi, gh1 = torch.empty_like(phi), torch.empty((sp.nk, sp.M, sp.M), dtype=torch.complex128, device="cuda")

    def backward(want_phi, want_h1):
        s = torch.cuda.current_stream().cuda_stream
        assert sys_.lib.afqmc_kp_local_energy_backward(sys_.handle, phi.data_ptr(), g.data_ptr(),
                                                       gphi.data_ptr() if want_phi else 0,
                                                       gh1.data_ptr() if want_h1 else 0, s) == 0

    calls = {
        "energy": lambda: sys_.local_energy(phi, eloc),
        "propagate": lambda: sys_.propagate(phi, x, w, logdet=ld),
        "step": lambda: sys_.step(phi, x, w, eloc, logdet=ld, do_qr=True, reuse=False),
        "orthonormalise": lambda: sys_.orthonormalise(phi, ld),
        "backward": lambda: backward(True, True),
        "backward, walkers": lambda: backward(True, False),
        "backward, one-body": lambda: backward(False, True),
    }
    for name, call in calls.items():
        nodes = kernel_nodes(call)
        assert sys_.launch_count() == nodes, name
    sys_.close()
