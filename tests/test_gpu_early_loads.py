"""Launches that start, or load, before the launch in front of them has ended: what they read is what their call's operands hold, and
the limit of their device-side waits does not count the time of the launch in front."""
import ctypes
import threading

import pytest
import torch

from paper_2309_03824_b200 import binding as b
from paper_2309_03824_b200 import workloads as wl

from helpers import TOL, dev, workspace

pytestmark = pytest.mark.gpu

HOLD = r"""
extern "C" __global__ void hold(int ms) {        // lets the next launch start, then keeps its one warp busy for ms
    asm volatile("griddepcontrol.launch_dependents;");
    unsigned long long t0, t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t0));
    t = t0;
    for (unsigned i = 0; i < 8000000u && t - t0 < ms * 1000000ull; ++i) {
        __nanosleep(1000);
        asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    }
}
"""


def test_a_long_launch_in_front_of_gradients():
    """Behind kernels of the caller that let their dependents start at once and run for longer than a device-side wait may last (17.2 s by
    the wait self-test): every form of a weight gradient, on a stream of its own."""
    kernel, ms = torch.cuda._compile_kernel(HOLD, "hold"), 22000
    M, K, N, r = 700, 264, 392, 72
    case = wl.random_factor_case(M, K, N, r, "bf16", 1100)
    desc = b.linear_desc(M, K, N, r, b.LRD_BF16)
    X, V, dY = (dev(case[k], "bf16") for k in ("X", "V", "dY"))
    Z = (X.float() @ V.float()).to(torch.bfloat16)
    B, H, W, C, S = 3, 9, 11, 40, 72
    Xc, dYc = (torch.randn(B, H, W, c, device="cuda").to(torch.bfloat16) for c in (C, S))
    Wk, dW = (torch.zeros(S, 3, 3, C, dtype=torch.bfloat16, device="cuda") for _ in range(2))
    ws_c = workspace(b.lrd_conv3x3_workspace_bytes(B, H, W, C, S, b.LRD_BF16))
    out = []
    torch.cuda.synchronize()
    b.lrd_check_device_status()
    try:
        for form in [(1, 128, 1), (1, 64, 4), (2, 256, 1)]:
            b.lrd_wgrad_tuning(*form)
            ws = workspace(b.lrd_linear_workspace_bytes(desc, b.LRD_FREEZE_V, 1))
            dU, db = torch.zeros(N, r, dtype=torch.bfloat16, device="cuda"), torch.zeros(N, dtype=torch.bfloat16, device="cuda")
            out.append((dU, db, ws))
            side = torch.cuda.Stream()
            side.wait_stream(torch.cuda.current_stream())
            with torch.cuda.stream(side):
                kernel((1, 1, 1), (32, 1, 1), [ms])
                b.lrd_linear_bwd_weights(desc, dY, None, Z, dU, None, db, b.LRD_FREEZE_V, ws)
    finally:
        b.lrd_wgrad_tuning()
    side = torch.cuda.Stream()
    with torch.cuda.stream(side):
        kernel((1, 1, 1), (32, 1, 1), [ms])
        b.lrd_conv3x3_bwd(B, H, W, C, S, b.LRD_BF16, dYc, Xc, Wk, None, dW, ws_c)
    assert b.lrd_check_device_status() == b.LRD_OK
    ref, sums = dY.double().T @ Z.double(), dY.double().sum(0)
    for dU, db, _ in out:                                               # (one rounding of the sums)
        assert float((dU.double() - ref).abs().max() / ref.abs().max()) <= 2 ** -8
        assert float((db.double() - sums).abs().max() / sums.abs().max()) <= 2 ** -8
    nchw = lambda t: t.double().permute(0, 3, 1, 2)
    ref = torch.nn.grad.conv2d_weight(nchw(Xc), (S, C, 3, 3), nchw(dYc), padding=1).permute(0, 2, 3, 1)
    assert float((dW.double() - ref).abs().max() / ref.abs().max()) <= 2 ** -8


def fresh_operands(bases, call, reference, ws, rounds=4):
    """Calls one after the other, each on operands that other kernels wrote right before it, in a workspace of NaN, and that are
    overwritten right behind it: what every call left is what the fp64 reference gives for its operands as they stood."""
    live = {k: torch.empty_like(v) for k, v in bases.items()}
    got = []
    for i in range(rounds):
        ws.view(torch.bfloat16).fill_(float("nan"))
        for j, (k, v) in enumerate(bases.items()):
            torch.mul(v, [1.0, -2.0, 0.5, 3.0][(i + j) % 4], out=live[k])
        got.append(call(live))
        for t in live.values():
            t.fill_(7.0 + i)
    torch.cuda.synchronize()
    assert b.lrd_check_device_status() == b.LRD_OK
    for i, out in enumerate(got):
        ref = reference({k: (v.float() * [1.0, -2.0, 0.5, 3.0][(i + j) % 4]).double() for j, (k, v) in enumerate(bases.items())})
        for k, t in out.items():
            if t is not None:
                assert float((t.double() - ref[k]).abs().max() / ref[k].abs().max()) <= TOL["bf16"], (i, k)


def linear_operands(M, K, N, r, seed, Z=False):
    case = wl.random_factor_case(M, K, N, r, "bf16", seed)
    t = {k: dev(case[k], "bf16") for k in ("X", "V", "dY", "b", "U")}
    return dict(t, Z=(t["X"].float() @ t["V"].float()).to(torch.bfloat16)) if Z else t


# tokens, K, N, r of the second product (its reduction): one k-block, a ring that is not filled, one that is, and is reused; several
# tiles a block; ranks whose rows are padded
@pytest.mark.parametrize("shape", [(200, 264, 520, 40), (300, 264, 520, 256), (700, 720, 776, 640), (2500, 264, 1032, 136), (9000, 136, 1032, 72), (64, 1096, 2056, 1024), (1021, 264, 520, 129)],
                         ids=lambda s: "x".join(map(str, s)))
@pytest.mark.parametrize("blocks", [1, 2])
@pytest.mark.parametrize("freeze", [b.LRD_FREEZE_U, b.LRD_FREEZE_V])
def test_the_second_factor_of_two_products(shape, blocks, freeze):
    M, K, N, r = shape
    desc = b.linear_desc(M, K, N, r, b.LRD_BF16)
    ws = workspace(b.lrd_linear_workspace_bytes(desc, freeze, 0))

    def call(t):
        out = {"Y": torch.empty_like(t["dY"]), "Z": None if freeze == b.LRD_FREEZE_U else torch.empty(M, r, dtype=torch.bfloat16, device="cuda")}
        b.lrd_linear_fwd(desc, t["X"], t["V"], t["U"], t["b"], out["Y"], out["Z"], freeze, ws)
        return out

    b.lrd_set_path(b.LRD_PATH_UNFUSED)
    b.lrd_gemm_tuning(blocks)
    try:
        fresh_operands(linear_operands(*shape, 1200 + M), call, lambda t: {"Z": t["X"] @ t["V"], "Y": (t["X"] @ t["V"]) @ t["U"].T + t["b"]}, ws)
    finally:
        b.lrd_set_path(b.LRD_PATH_AUTO)
        b.lrd_gemm_tuning(0)


def linear_gradients(t, add=0.0):
    dZ = t["dY"] @ t["U"]
    return {"dX": dZ @ t["V"].T, "dU": t["dY"].T @ t["Z"] + add, "dV": t["X"].T @ dZ + add, "db": t["dY"].sum(0) + add}


@pytest.mark.parametrize("freeze", [b.LRD_FREEZE_V, b.LRD_FREEZE_U, b.LRD_FREEZE_NONE])
@pytest.mark.parametrize("shape", [(4096, 768, 768, 192), (128, 768, 768, 192), (1021, 1024, 1024, 512), (300, 520, 520, 250), (2000, 264, 264, 64), (2048, 1024, 2056, 250)],
                         ids=lambda s: "x".join(map(str, s)))
@pytest.mark.parametrize("path", [b.LRD_PATH_AUTO, b.LRD_PATH_UNFUSED])
@pytest.mark.parametrize("adding", [False, True])
def test_the_gradients_of_a_layer(shape, freeze, path, adding):
    """What dU, dV and the second factor of the data pass load ahead; adding, to what an earlier launch left in the caller's buffers."""
    M, K, N, r = shape
    desc = b.linear_desc(M, K, N, r, b.LRD_BF16)
    ws = workspace(b.lrd_linear_workspace_bytes(desc, freeze, 2 if adding else 1))
    backward = b.lrd_linear_bwd_accumulate if adding else b.lrd_linear_bwd

    def call(t):
        out = {k: torch.full(s, 2.0 if adding else float("nan"), dtype=torch.bfloat16, device="cuda") for k, s in (("dU", (N, r)), ("dV", (K, r)), ("db", (N,)))}
        if freeze == b.LRD_FREEZE_U:
            out.update(dU=None, db=None)
        if freeze == b.LRD_FREEZE_V:
            out.update(dV=None)
        out["dX"] = torch.empty_like(t["X"])
        backward(desc, t["dY"], t["X"], t["V"], t["U"], t["Z"], out["dX"], out["dU"], out["dV"], out["db"], freeze, ws)
        return out

    b.lrd_set_path(path)
    try:
        fresh_operands(linear_operands(*shape, 1300 + M, Z=True), call, lambda t: linear_gradients(t, 2.0 if adding else 0.0), ws)
    finally:
        b.lrd_set_path(b.LRD_PATH_AUTO)


MASKS = [b.LRD_TK_FREEZE_NONE, b.LRD_TK_FREEZE_FACTORS, b.LRD_TK_FREEZE_CORE]
# whole pass in one launch; 1x1 products apart from the core, then (S > 256) the last one too; the same at ranks whose rows are padded;
# stride 2 with the core and one product in a launch, then apart, then padded
CONVS = [(16, 14, 14, 64, 72, 32, 48, 3, 1), (8, 9, 11, 136, 128, 96, 104, 3, 1), (16, 7, 7, 264, 272, 136, 144, 3, 1), (16, 7, 7, 264, 272, 135, 141, 3, 1),
         (8, 14, 14, 72, 136, 48, 48, 3, 2), (16, 13, 14, 264, 272, 136, 152, 3, 2), (16, 14, 13, 264, 272, 130, 150, 3, 2), (8, 9, 9, 40, 264, 24, 40, 5, 1)]


def conv_layer(t, stride):
    nchw = lambda x: x.permute(0, 3, 1, 2)
    Z1 = t["X"] @ t["A"]
    Z2 = torch.nn.functional.conv2d(nchw(Z1), t["G"].permute(0, 3, 1, 2), stride=stride, padding=t["G"].shape[1] // 2).permute(0, 2, 3, 1)
    return Z1, Z2, Z2 @ t["Bm"].T + t["b"]


def conv_operands(geom, seed):
    B, H, W, C, S, r1, r2, k, stride = geom
    case = wl.random_tucker_case(B, H, W, C, S, r1, r2, k, "bf16", seed, stride=stride)
    return {n: dev(case[n], "bf16") for n in ("X", "A", "G", "Bm", "b", "dY")}


@pytest.mark.parametrize("geom", CONVS, ids=lambda g: "x".join(map(str, g)))
@pytest.mark.parametrize("freeze", MASKS)
def test_the_second_factor_and_the_copies_of_a_convolution(geom, freeze):
    """The forward pass: the last product's factor, and Z1 and Z2 copied to the caller's rows beside it."""
    B, H, W, C, S, r1, r2, k, stride = geom
    desc = b.tucker2_desc(B, H, W, C, S, r1, r2, b.LRD_BF16, k=k, stride=stride, pad=(k - 1) // 2)
    ws = workspace(b.lrd_tucker2_workspace_bytes(desc, freeze, 0))
    Ho, Wo = (H - 1) // stride + 1, (W - 1) // stride + 1

    def call(t):
        new = lambda *s: torch.empty(*s, dtype=torch.bfloat16, device="cuda")
        out = {"Y": new(B, Ho, Wo, S), "Z1": None if freeze == b.LRD_TK_FREEZE_CORE else new(B, H, W, r1), "Z2": None if freeze == b.LRD_TK_FREEZE_FACTORS else new(B, Ho, Wo, r2)}
        b.lrd_tucker2_fwd(desc, t["X"], t["A"], t["G"], t["Bm"], t["b"], out["Y"], out["Z1"], out["Z2"], freeze, ws)
        return out

    fresh_operands(conv_operands(geom, 1400 + C), call, lambda t: dict(zip(("Z1", "Z2", "Y"), conv_layer(t, stride))), ws)


@pytest.mark.parametrize("geom", CONVS, ids=lambda g: "x".join(map(str, g)))
@pytest.mark.parametrize("freeze", MASKS)
@pytest.mark.parametrize("overlap", [True, False])
def test_the_gradients_of_a_convolution(geom, freeze, overlap):
    """dA and dB with the core frozen, the filter gradient that follows the data path or runs beside it, the last product's factor."""
    B, H, W, C, S, r1, r2, k, stride = geom
    desc = b.tucker2_desc(B, H, W, C, S, r1, r2, b.LRD_BF16, k=k, stride=stride, pad=(k - 1) // 2)
    ws = workspace(b.lrd_tucker2_workspace_bytes(desc, freeze, 1))
    bases = conv_operands(geom, 1500 + C)
    with torch.no_grad():
        Z1, Z2, _ = conv_layer({n: v.double() for n, v in bases.items()}, stride)
    bases.update(Z1=Z1.to(torch.bfloat16).contiguous(), Z2=Z2.to(torch.bfloat16).contiguous())
    factors, core = freeze != b.LRD_TK_FREEZE_FACTORS, freeze != b.LRD_TK_FREEZE_CORE

    def call(t):
        out = {"dX": torch.empty_like(t["X"]), "dA": torch.empty_like(t["A"]) if factors else None, "dB": torch.empty_like(t["Bm"]) if factors else None,
               "db": torch.empty_like(t["b"]) if factors else None, "dG": torch.empty_like(t["G"]) if core else None}
        b.lrd_tucker2_bwd(desc, t["dY"], t["X"] if factors else None, t["A"], t["G"], t["Bm"], t["Z1"] if core else None, t["Z2"] if factors else None, out["dX"],
                          out["dA"], out["dG"], out["dB"], out["db"], freeze, ws)
        return out

    def reference(t):
        nchw = lambda x: x.permute(0, 3, 1, 2)
        G, pad = nchw(t["G"]), k // 2
        dZ2 = t["dY"] @ t["Bm"]
        dZ1 = torch.nn.grad.conv2d_input((B, r1, H, W), G, nchw(dZ2), stride=stride, padding=pad).permute(0, 2, 3, 1)
        dG = torch.nn.grad.conv2d_weight(nchw(t["Z1"]), G.shape, nchw(dZ2), stride=stride, padding=pad).permute(0, 2, 3, 1)
        flat = lambda x: x.reshape(-1, x.shape[-1])
        return {"dX": dZ1 @ t["A"].T, "dA": flat(t["X"]).T @ flat(dZ1), "dB": flat(t["dY"]).T @ flat(t["Z2"]), "db": flat(t["dY"]).sum(0), "dG": dG}

    b.lrd_tucker2_overlap(overlap)
    try:
        fresh_operands(bases, call, reference, ws)
    finally:
        b.lrd_tucker2_overlap(True)


class Edge(ctypes.Structure):
    _fields_ = [("from_port", ctypes.c_ubyte), ("to_port", ctypes.c_ubyte), ("type", ctypes.c_ubyte), ("reserved", ctypes.c_ubyte * 5)]


def branches(graph):
    """Launches of a captured graph that more than one other follows."""
    cu, count = ctypes.CDLL("libcuda.so.1"), ctypes.c_size_t(64)
    ends, edges = [(ctypes.c_void_p * 64)() for _ in range(2)], (Edge * 64)()
    assert cu.cuGraphGetEdges_v2(ctypes.c_void_p(graph.raw_cuda_graph()), ends[0], ends[1], edges, ctypes.byref(count)) == 0
    froms = ends[0][:count.value]
    return sum(froms.count(n) > 1 for n in set(froms))


# the core's data gradient on few blocks; on as many as there are SMs; the whole data path in one launch
@pytest.mark.parametrize("geom,beside", [((16, 7, 7, 264, 272, 136, 144, 3, 1), True), ((8, 14, 14, 72, 136, 48, 48, 3, 2), True), ((64, 14, 14, 264, 272, 320, 256, 3, 1), False),
                                         ((16, 14, 14, 64, 72, 32, 48, 3, 1), False)], ids=lambda g: str(g))
def test_a_captured_filter_gradient_runs_beside_a_data_path_that_leaves_it_room(geom, beside):
    """With the factors frozen: beside the data path in a graph, behind it elsewhere and where a thread's first call is captured (it has no
    streams then); the same bits each way."""
    B, H, W, C, S, r1, r2, k, stride = geom
    r1, r2 = min(r1, C), min(r2, S)
    freeze = b.LRD_TK_FREEZE_FACTORS
    desc = b.tucker2_desc(B, H, W, C, S, r1, r2, b.LRD_BF16, k=k, stride=stride, pad=(k - 1) // 2)
    t = conv_operands((B, H, W, C, S, r1, r2, k, stride), 1600 + B)
    Z1 = (t["X"].float() @ t["A"].float()).to(torch.bfloat16)
    ws = workspace(b.lrd_tucker2_workspace_bytes(desc, freeze, 1))
    dX, dG = torch.empty_like(t["X"]), torch.empty_like(t["G"])
    call = lambda: b.lrd_tucker2_bwd(desc, t["dY"], None, t["A"], t["G"], t["Bm"], Z1, None, dX, None, dG, None, None, freeze, ws)
    call()
    torch.cuda.synchronize()
    want = dX.clone(), dG.clone()
    found = []

    def capture():
        side, graph = torch.cuda.Stream(), torch.cuda.CUDAGraph(keep_graph=True)
        with torch.cuda.stream(side), torch.cuda.graph(graph, stream=side, capture_error_mode="thread_local"):
            call()
        dX.zero_()
        dG.zero_()
        torch.cuda.synchronize()
        graph.replay()
        torch.cuda.synchronize()
        found.append((branches(graph), torch.equal(dX, want[0]), torch.equal(dG, want[1])))

    capture()
    other = threading.Thread(target=capture)
    other.start()
    other.join()
    assert found == [(1 if beside else 0, True, True), (0, True, True)]
    assert b.lrd_check_device_status() == b.LRD_OK
