"""Launches that start, or load, before the launch in front of them has ended: what they read is what their call's operands hold, and
the limit of their device-side waits does not count the time of the launch in front."""
import pytest
import torch

from paper_2309_03824_b200 import binding as b
from paper_2309_03824_b200 import workloads as wl

from helpers import dev, workspace

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
