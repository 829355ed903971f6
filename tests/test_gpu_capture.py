"""GPU: calls captured into a CUDA graph. Nothing orders a graph's nodes, or its replays,
against other calls on the context, so calls that shared nothing with others take no scratch
of it: two on parallel branches give the bits of the same calls alone.
"""
import ctypes

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

KERNEL_NODE = 0  # cudaGraphNodeTypeKernel


@pytest.fixture(scope="module")
def rt():
    lib = ctypes.CDLL("libcudart.so.13")
    vp = ctypes.c_void_p
    lib.cudaStreamBeginCapture.argtypes = [vp, ctypes.c_int]
    lib.cudaStreamEndCapture.argtypes = [vp, ctypes.POINTER(vp)]
    lib.cudaGraphGetNodes.argtypes = [vp, ctypes.POINTER(vp), ctypes.POINTER(ctypes.c_size_t)]
    lib.cudaGraphNodeGetType.argtypes = [vp, ctypes.POINTER(ctypes.c_int)]
    lib.cudaGraphInstantiate.argtypes = [ctypes.POINTER(vp), vp, ctypes.c_ulonglong]
    lib.cudaGraphLaunch.argtypes = [vp, vp]
    lib.cudaGraphExecDestroy.argtypes = [vp]
    lib.cudaGraphDestroy.argtypes = [vp]
    return lib


def capture(rt, stream, calls):
    """The graph of calls() on the stream, and its number of kernels."""
    import torch
    torch.cuda.synchronize()
    graph = ctypes.c_void_p()
    assert rt.cudaStreamBeginCapture(stream.cuda_stream, 2) == 0  # relaxed
    try:
        calls()
    finally:
        assert rt.cudaStreamEndCapture(stream.cuda_stream, ctypes.byref(graph)) == 0
    n = ctypes.c_size_t()
    assert rt.cudaGraphGetNodes(graph, None, ctypes.byref(n)) == 0
    nodes = (ctypes.c_void_p * n.value)()
    assert rt.cudaGraphGetNodes(graph, nodes, ctypes.byref(n)) == 0
    kinds = []
    for node in nodes:
        kind = ctypes.c_int()
        assert rt.cudaGraphNodeGetType(node, ctypes.byref(kind)) == 0
        kinds.append(kind.value)
    return graph, kinds.count(KERNEL_NODE)


def replay(rt, graph, stream, times=3):
    import torch
    run = ctypes.c_void_p()
    assert rt.cudaGraphInstantiate(ctypes.byref(run), graph, 0) == 0
    for _ in range(times):
        assert rt.cudaGraphLaunch(run, stream.cuda_stream) == 0
    torch.cuda.synchronize()
    assert rt.cudaGraphExecDestroy(run) == 0
    assert rt.cudaGraphDestroy(graph) == 0


def on_two_branches(stream, other, a, b):
    """a() on the stream beside b() on the other one, joined again."""
    import torch
    fork, join = torch.cuda.Event(), torch.cuda.Event()
    fork.record(stream)
    other.wait_event(fork)
    a()
    b()
    join.record(other)
    stream.wait_event(join)


def sparse_planes(b, n_rot, n_data, precision, seed):
    """P with a handful of non-zero frames a row, as emc_update takes it."""
    import torch
    g = torch.Generator(device="cuda").manual_seed(seed)
    P = torch.zeros((b.rows, b.ld_data), device="cuda")
    rows = torch.arange(n_rot, device="cuda")
    for _ in range(3):
        k = torch.randint(n_data, (n_rot,), generator=g, device="cuda")
        P[rows, k] = 0.1 + torch.rand(n_rot, generator=g, device="cuda")
    if precision != "fp32":
        hi = P.to(torch.bfloat16)
        P = torch.stack([hi, (P - hi.float()).to(torch.bfloat16)])
    return P.contiguous()


@pytest.mark.parametrize("precision", ["fp32", "bf16_split"])
def test_captured_updates_share_nothing(rt, precision):
    import torch
    from paper_1409_4256_gb300 import emc, synth
    det = synth.make_detector(60, 16)
    quat, w = emc.quat_generate(4)
    n_rot, n_data = quat.shape[0], 5300
    ctx = emc.Context(16, det.q, quat, w, n_data, precision=precision)
    K = np.random.default_rng(8).poisson(0.7, size=(n_data, det.q.shape[0])).astype(np.int32)
    ctx.set_frames(torch.as_tensor(K, device="cuda"))
    b = ctx.buffer_sizes(n_rot)
    P = [sparse_planes(b, n_rot, n_data, precision, s) for s in (1, 2)]
    Num = [torch.empty((b.rows, b.ld_pix), device="cuda") for _ in P]
    den = [torch.empty(b.rows, device="cuda") for _ in P]
    streams = [torch.cuda.Stream(), torch.cuda.Stream()]

    def update(i):
        emc._check(emc.lib().emc_update(ctx.h, P[i].data_ptr(), n_rot, Num[i].data_ptr(),
                                        den[i].data_ptr(), streams[i].cuda_stream), "emc_update")

    want = []
    for i in (0, 1):  # alone in a graph each: every frame contracted, in order
        graph, kernels = capture(rt, streams[i], lambda: update(i))
        assert kernels == 1
        replay(rt, graph, streams[i], 1)
        want.append((Num[i].clone(), den[i].clone()))
        eager, eden = ctx.update(P[i], n_rot)
        # FP32 order, 3 products of one sign a row at most (split: hi and lo ones)
        assert torch.allclose(eager[:n_rot], Num[i][:n_rot], rtol=8 * 2.0 ** -23, atol=0)
        assert torch.allclose(eden[:n_rot], den[i][:n_rot], rtol=8 * 2.0 ** -23, atol=0)
    graph, kernels = capture(rt, streams[0], lambda: on_two_branches(
        streams[0], streams[1], lambda: update(0), lambda: update(1)))
    assert kernels == 2
    for i in (0, 1):
        Num[i].zero_()
        den[i].zero_()
    replay(rt, graph, streams[0])
    for i in (0, 1):
        assert torch.equal(Num[i], want[i][0]) and torch.equal(den[i], want[i][1])
    assert ctx.status() == 0


def test_fluence_expansion_takes_no_scratch(rt):
    """The Poisson-fluence expansion keeps W and its sums in the caller's L on the way: of the
    context's workspace a call writes its rotations' B_j alone (pixels at the grid's edge, so
    without the cell layout of the model), and two captured ones on parallel branches, each
    with a model and a block of its own, give the bits of the calls alone."""
    import torch
    from paper_1409_4256_gb300 import emc, synth
    det = synth.make_detector(40, 32)
    q = det.q * (15.99 / 15.0)
    quat, w = emc.quat_generate(4)
    n = quat.shape[0]
    ctx = emc.Context(32, q, quat, w, 300, model="poisson_fluence", w_floor=1e-6)
    ctx.set_frames(torch.ones(300, q.shape[0], dtype=torch.int32, device="cuda"))
    g = torch.Generator(device="cuda").manual_seed(3)
    grids = [torch.rand(32, 32, 32, generator=g, device="cuda") + 0.1 for _ in range(2)]
    blocks = [(0, 1280), (1280, n - 1280)]
    out = []
    for r0, nb in blocks:
        b = ctx.buffer_sizes(nb)
        out.append((torch.empty(b.logw_bytes, dtype=torch.uint8, device="cuda"),
                    torch.empty(b.bias_bytes // 8, dtype=torch.float64, device="cuda")))
    streams = [torch.cuda.Stream() for _ in range(2)]

    def expand(i):
        emc._check(emc.lib().emc_expand(ctx.h, grids[i].data_ptr(), *blocks[i],
                                        out[i][0].data_ptr(), out[i][1].data_ptr(),
                                        streams[i].cuda_stream), "emc_expand")

    want = []
    for i in (0, 1):
        torch.cuda.synchronize()
        before = ctx.workspace.clone()
        torch.cuda.synchronize()
        expand(i)
        torch.cuda.synchronize()
        changed = torch.nonzero(ctx.workspace != before)
        assert int(changed.amax() - changed.amin()) < 8 * ctx.buffer_sizes(blocks[i][1]).rows
        want.append([x.clone() for x in out[i]])
    graph, _ = capture(rt, streams[0], lambda: on_two_branches(
        streams[0], streams[1], lambda: expand(0), lambda: expand(1)))
    for x in out:
        x[0].zero_()
        x[1].zero_()
    replay(rt, graph, streams[0])
    for i in (0, 1):
        assert torch.equal(out[i][0], want[i][0]) and torch.equal(out[i][1], want[i][1])
    assert ctx.status() == 0
