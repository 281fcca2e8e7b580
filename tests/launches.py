"""The kernel launches of a call, read from a stream capture (nothing runs), and a
call's device time."""
import ctypes
from dataclasses import dataclass

import torch

RELAXED = 2          # CU_STREAM_CAPTURE_MODE_RELAXED
KERNEL_NODE = 0      # CU_GRAPH_NODE_TYPE_KERNEL


class _Params(ctypes.Structure):   # CUDA_KERNEL_NODE_PARAMS_v2
    _fields_ = [("func", ctypes.c_void_p), ("grid", ctypes.c_uint * 3),
                ("block", ctypes.c_uint * 3), ("smem", ctypes.c_uint),
                ("params", ctypes.c_void_p), ("extra", ctypes.c_void_p),
                ("kern", ctypes.c_void_p), ("ctx", ctypes.c_void_p)]


@dataclass
class Launch:
    name: str
    ctas: int
    threads: int
    per_sm: int      # CTAs that fit on an SM

    @property
    def resident(self):
        return self.per_sm * torch.cuda.get_device_properties(0).multi_processor_count


def launches(call):
    """[Launch] of ``call(stream)``, in no particular order."""
    cu = ctypes.CDLL("libcuda.so.1")

    def do(name, *args):
        status = getattr(cu, name)(*args)
        assert status == 0, (name, status)

    torch.cuda.init()
    stream = torch.cuda.Stream()
    h = ctypes.c_void_p(stream.cuda_stream)
    graph = ctypes.c_void_p()
    do("cuStreamBeginCapture_v2", h, RELAXED)
    try:
        call(stream)
    finally:
        do("cuStreamEndCapture", h, ctypes.byref(graph))
    n = ctypes.c_size_t()
    do("cuGraphGetNodes", graph, None, ctypes.byref(n))
    nodes = (ctypes.c_void_p * n.value)()
    do("cuGraphGetNodes", graph, nodes, ctypes.byref(n))
    found = []
    for node in nodes:
        node = ctypes.c_void_p(node)
        kind = ctypes.c_int()
        do("cuGraphNodeGetType", node, ctypes.byref(kind))
        if kind.value != KERNEL_NODE:
            continue
        p = _Params()
        do("cuGraphKernelNodeGetParams_v2", node, ctypes.byref(p))
        func = ctypes.c_void_p(p.func)
        if not func:
            do("cuKernelGetFunction", ctypes.byref(func), ctypes.c_void_p(p.kern))
        name = ctypes.c_char_p()
        do("cuFuncGetName", ctypes.byref(name), func)
        threads = p.block[0] * p.block[1] * p.block[2]
        per_sm = ctypes.c_int()
        do("cuOccupancyMaxActiveBlocksPerMultiprocessor", ctypes.byref(per_sm), func, threads,
           ctypes.c_size_t(p.smem))
        found.append(Launch(name.value.decode(), p.grid[0] * p.grid[1] * p.grid[2], threads,
                            per_sm.value))
    do("cuGraphDestroy", graph)
    return found


def device_us(call, calls=12, replays=20):
    """Device time of ``call()`` among others of its kind: the least over replays of a
    graph of them (what else runs on the machine can only add to it)."""
    call()
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        for _ in range(calls):
            call()
    times = []
    for _ in range(5 + replays):
        start, end = (torch.cuda.Event(enable_timing=True) for _ in range(2))
        start.record()
        graph.replay()
        end.record()
        end.synchronize()
        times.append(start.elapsed_time(end) * 1e3 / calls)
    return min(times[5:])
