"""Which calls may start before the kernel ahead of them has ended, read from the edges of captured graphs: a GEMV or GEMM directly
behind the device packer may not (it reads packed weights before it waits), one behind another GEMV or GEMM may."""
import ctypes

import numpy as np
import pytest
import torch

import gpu_util as gu
from paper_2606_11357_b200 import binding as tf
from paper_2606_11357_b200 import workloads as wl

pytestmark = pytest.mark.gpu

K, N = 1024, 1032


class Calls:
    def __init__(self):
        self.problem = wl.make_w4(40, K, N, seed=70)
        p = self.problem
        self.arrays = [torch.from_numpy(p.qweight.view(np.int32)).cuda(), torch.from_numpy(p.scales_f16).cuda(), torch.from_numpy(p.qzeros.view(np.int32)).cuda()]
        self.blob = torch.from_numpy(gu.pack(p)).cuda()
        self.a = gu.to_device_bf16(p.a_bf16)
        self.y = torch.zeros(40, N, dtype=torch.bfloat16, device="cuda")
        self.ws = torch.zeros(tf.tf_workspace_size(tf.TF_OP_GEMM_W4A16, 40, K, N), dtype=torch.uint8, device="cuda")

    def __call__(self, letter):
        if letter == "p":
            tf.tf_pack_awq_device(*self.arrays, K, N, 128, self.blob)
        elif letter == "g":
            tf.tf_gemm_w4a16(self.blob, self.a, self.y, 40, K, N, self.ws)
        else:
            tf.tf_gemv_w4a16(self.blob, self.a[:int(letter)], self.y[:int(letter)], int(letter), K, N, self.ws)


def capture(body):
    graph = torch.cuda.CUDAGraph(keep_graph=True)
    with torch.cuda.graph(graph):
        body()
    return graph


class EdgeData(ctypes.Structure):                               # cudaGraphEdgeData
    _fields_ = [("from_port", ctypes.c_ubyte), ("to_port", ctypes.c_ubyte), ("type", ctypes.c_ubyte), ("reserved", ctypes.c_ubyte * 5)]


def edges(graph):
    """{(from, to): may the second start early}, the nodes as the handles' values."""
    get = ctypes.CDLL("libcudart.so.12").cudaGraphGetEdges_v2   # (torch has loaded it)
    handle, count = ctypes.c_void_p(graph.raw_cuda_graph()), ctypes.c_size_t(0)
    assert get(handle, None, None, None, ctypes.byref(count)) == 0
    begin, end, data = ((t * count.value)() for t in (ctypes.c_void_p, ctypes.c_void_p, EdgeData))
    assert get(handle, begin, end, data, ctypes.byref(count)) == 0
    return {(b, e): d.type == 1 for b, e, d in zip(begin, end, data)}       # 1: cudaGraphDependencyTypeProgrammatic


def in_order(links):
    """The answers along a graph that is one chain."""
    then = {b: (e, early) for (b, e), early in links.items()}
    (node,) = set(then) - {e for e, _ in then.values()}
    out = []
    while node in then:
        node, early = then[node]
        out.append(early)
    assert len(out) == len(links)
    return out


# a digit: a GEMV of that many tokens; g: a GEMM; p: the packer (which waits itself, so it may start early behind anything that lets it)
@pytest.mark.parametrize("calls,late", [("114g9", ()), ("1p1p4pgp", (2, 4, 6)), ("p11p", (1,)), ("gppg1", (2, 3))])
def test_calls_directly_behind_the_packer_are_ordinary_launches(calls, late):
    c = Calls()
    for letter in calls:                                         # set-up of the library; and notes that a capture must not go by
        c(letter)
    c("1")
    graph = capture(lambda: [c(letter) for letter in calls])
    answers = in_order(edges(graph))
    for i, letter in enumerate(calls[1:], 1):
        if letter != "p":
            assert answers[i - 1] == (i not in late), (calls, i)


def test_packing_on_another_stream_of_a_capture():
    """A second stream waits for the packer by an event, after a GEMV of its own: no edge out of the packer lets its dependent start early."""
    c = Calls()
    for letter in "1p4":
        c(letter)
    side = torch.cuda.Stream()

    def body():
        main = torch.cuda.current_stream()
        c("1")
        side.wait_stream(main)
        with torch.cuda.stream(side):
            c("4")
        main.wait_stream(side)
        c("p")
        side.wait_stream(main)
        with torch.cuda.stream(side):
            c("4")
            c("1")
        main.wait_stream(side)

    links = edges(capture(body))
    (last,) = {e for _, e in links} - {b for b, _ in links}
    (reader,) = {b for b, e in links if e == last}
    into_reader = {b: early for (b, e), early in links.items() if e == reader}
    assert into_reader and not any(into_reader.values())
    assert links[(reader, last)]


def test_a_packing_is_remembered_while_many_other_streams_launch():
    """On the running stream: packing, then calls on more streams than are remembered, then the call that reads the blob."""
    c = Calls()
    c("1")
    blob, streams = c.blob.clone(), [torch.cuda.Stream() for _ in range(40)]
    others = [(torch.zeros(1, N, dtype=torch.bfloat16, device="cuda"), torch.zeros_like(c.ws)) for _ in streams]
    torch.cuda.synchronize()
    for rep in range(3):
        c.blob.zero_()
        c.y.fill_(float("nan"))
        c("p")
        for s, (y, ws) in zip(streams, others):
            with torch.cuda.stream(s):
                tf.tf_gemv_w4a16(blob, c.a[:1], y, 1, K, N, ws)
        c("g")
        assert tf.tf_device_status(c.ws) == 0
        gu.check_against_oracle(c.problem, gu.bits_of(c.y))
        torch.cuda.synchronize()
        assert all(torch.equal(y, others[0][0]) for y, _ in others)
