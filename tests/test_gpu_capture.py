"""sg_matvec under stream capture: the graph is made of kernels alone, so that it can be instantiated
more than once and be a child graph, and its scratch lives as long as it does."""

import ctypes
import time

import pytest

from paper_1910_11505_gb300 import sg, workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


class _Graphs:
    """The CUDA runtime's graph calls; every error code raises."""

    def __init__(self):
        for name in ("libcudart.so.13", "/usr/local/cuda/lib64/libcudart.so"):
            try:
                self.rt = ctypes.CDLL(name)
                break
            except OSError:
                pass

    def __getattr__(self, name):
        def call(*args):
            rc = getattr(self.rt, name)(*args)
            assert rc == 0, (name, rc)
        return call

    def capture(self, stream, body):
        g = ctypes.c_void_p()
        self.cudaStreamBeginCapture(ctypes.c_void_p(stream.cuda_stream), 1)
        body()
        self.cudaStreamEndCapture(ctypes.c_void_p(stream.cuda_stream), ctypes.byref(g))
        return g

    def instance(self, graph):
        e = ctypes.c_void_p()
        self.cudaGraphInstantiate(ctypes.byref(e), graph, ctypes.c_ulonglong(0))
        return e

    def launch(self, e, stream):
        self.cudaGraphLaunch(e, ctypes.c_void_p(stream.cuda_stream))

    def kinds(self, graph):
        n = ctypes.c_size_t()
        self.cudaGraphGetNodes(graph, None, ctypes.byref(n))
        nodes = (ctypes.c_void_p * n.value)()
        self.cudaGraphGetNodes(graph, nodes, ctypes.byref(n))
        out = []
        for node in nodes:
            t = ctypes.c_int()
            self.cudaGraphNodeGetType(ctypes.c_void_p(node), ctypes.byref(t))
            out.append(t.value)
        return out


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
def test_captured_operator_instances_and_child_graphs(precision):
    h = sg.sg_setup(sg.sg_default_params(n=64, M=4, p=3, sigma=0.8, ell=0.6, precision=precision))
    assert sg.sg_op_info(h)[precision]["kernel"] == "block"
    N, P, _ = sg.sg_dims(h)
    dt = torch.float64 if precision == "fp64" else torch.float32
    apply = sg.sg_matvec if precision == "fp64" else sg.sg_matvec_lowp
    X = torch.from_numpy(W.random_field(N, P, seed=1)).cuda().to(dt)
    want = [torch.empty_like(X) for _ in range(2)]
    apply(h, 0, X, want[0])
    apply(h, 0, want[0], want[1])
    Y = [torch.empty_like(X) for _ in range(2)]
    rt, s, s2 = _Graphs(), torch.cuda.Stream(), torch.cuda.Stream()
    torch.cuda.synchronize()

    def body():
        apply(h, 0, X, Y[0], stream=s)
        apply(h, 0, Y[0], Y[1], stream=s)

    def check(*launches):
        for y in Y:
            y.fill_(float("nan"))
        torch.cuda.synchronize()
        for e, st in launches:
            rt.launch(e, st)
        torch.cuda.synchronize()
        assert torch.equal(Y[0], want[0]) and torch.equal(Y[1], want[1])

    g = rt.capture(s, body)
    assert rt.kinds(g) == [0, 0, 0, 0]  # kernel nodes
    one, two = rt.instance(g), rt.instance(g)
    check((one, s))
    check((two, s2))
    check((one, s), (two, s2))  # both at once: the same values to the same places
    parent, node = ctypes.c_void_p(), ctypes.c_void_p()
    rt.cudaGraphCreate(ctypes.byref(parent), 0)
    rt.cudaGraphAddChildGraphNode(ctypes.byref(node), parent, None, ctypes.c_size_t(0), g)
    whole = rt.instance(parent)
    check((whole, s))
    # two streams of one capture
    both = [torch.empty_like(X), torch.empty_like(X)]

    def fork():
        s2.wait_stream(s)
        apply(h, 0, X, both[0], stream=s)
        apply(h, 0, want[0], both[1], stream=s2)
        s.wait_stream(s2)

    gf = rt.capture(s, fork)
    ef = rt.instance(gf)
    for _ in range(10):
        rt.launch(ef, s)
    torch.cuda.synchronize()
    assert torch.equal(both[0], want[0]) and torch.equal(both[1], want[1])
    rt.cudaGraphDestroy(g)
    check((one, s))  # an instance keeps the scratch
    for e in (one, two, whole, ef):
        rt.cudaGraphExecDestroy(e)
    for graph in (parent, gf):
        rt.cudaGraphDestroy(graph)
    # blocks of destroyed graphs serve the next ones
    free0 = torch.cuda.mem_get_info()[0]
    for _ in range(50):
        time.sleep(0.002)
        g = rt.capture(s, body)
        rt.cudaGraphDestroy(g)
    assert free0 - torch.cuda.mem_get_info()[0] <= 4 * 5 * N * P * X.element_size()
    h.close()


def test_graph_destroyed_after_its_handle():
    h = sg.sg_setup(sg.sg_default_params(n=64, M=4, p=3, sigma=0.8, ell=0.6))
    N, P, _ = sg.sg_dims(h)
    X = torch.zeros(N, P, dtype=torch.float64, device="cuda")
    Y, s, rt = torch.empty_like(X), torch.cuda.Stream(), _Graphs()
    torch.cuda.synchronize()
    g = rt.capture(s, lambda: sg.sg_matvec(h, 0, X, Y, stream=s))
    h.close()
    rt.cudaGraphDestroy(g)
    time.sleep(0.01)
