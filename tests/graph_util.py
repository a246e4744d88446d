"""What a call queues on a stream: its work captured into a CUDA graph through
the driver API, the graph's kernel launches counted."""
import ctypes as C


def kernels_of(stream, call):
    """Kernel launches that `call` queues on the stream handle (nothing runs)."""
    cu = C.CDLL("libcuda.so.1")

    def ck(r):
        assert r == 0, f"CUDA driver error {r}"

    st, graph, n = C.c_void_p(stream), C.c_void_p(), C.c_size_t()
    ck(cu.cuStreamBeginCapture_v2(st, 1))  # thread-local
    try:
        call()
    finally:
        r = cu.cuStreamEndCapture(st, C.byref(graph))
    ck(r)
    ck(cu.cuGraphGetNodes(graph, None, C.byref(n)))
    nodes = (C.c_void_p * n.value)()
    ck(cu.cuGraphGetNodes(graph, nodes, C.byref(n)))
    count = 0
    for x in nodes:
        t = C.c_int()
        ck(cu.cuGraphNodeGetType(C.c_void_p(x), C.byref(t)))
        count += t.value == 0
    ck(cu.cuGraphDestroy(graph))
    return count
