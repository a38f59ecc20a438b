"""Weight gradients of one backward pass in one launch: each tile width, single blocks, clusters and pairs of SMs, products of
different heights (rows past one product belong to the next), ranks that end inside a tile, with and without the bias gradient."""
import pytest
import torch

from paper_2309_03824_b200 import binding as b
from paper_2309_03824_b200 import workloads as wl

from helpers import check_linear, rel_err, run_linear

pytestmark = pytest.mark.gpu

# tokens, K, N, r; what the estimates choose, when this was written (width, blocks per tile): 192 x 2, 192 x 1, 64 x 1, 192 x 8, 64 x 4,
# 128 x 1, 128 x 8, 64 x 8, pairs 256 wide (every form by name: test_gpu_forms.py)
SHAPES = [(4096, 768, 3072, 384), (1024, 1024, 4096, 520), (70, 264, 200, 56), (5000, 520, 1000, 136), (2000, 264, 520, 248),
          (70, 1000, 4096, 200), (9000, 264, 520, 72), (9000, 264, 392, 40), (70, 4096, 4096, 504)]


@pytest.mark.parametrize("shape", SHAPES, ids=["x".join(map(str, s)) for s in SHAPES])
def test_both_factors(shape):
    case = wl.random_factor_case(*shape, "bf16", 900 + shape[0])
    got, _ = check_linear(case, b.LRD_FREEZE_NONE)
    again = run_linear(case, b.LRD_FREEZE_NONE)
    M, K, N, r = shape
    desc = b.linear_desc(M, K, N, r, b.LRD_BF16)
    X, dY, V, U = (torch.from_numpy(case[k]).to("cuda", torch.bfloat16) for k in ("X", "dY", "V", "U"))
    dX, dU, dV = torch.empty_like(X), torch.empty_like(got["dU"]), torch.empty_like(got["dV"])
    ws = torch.empty(b.lrd_linear_workspace_bytes(desc, b.LRD_FREEZE_NONE, 1), dtype=torch.uint8, device="cuda")
    b.lrd_linear_bwd(desc, dY, X, V, U, got["Z"], dX, dU, dV, None, b.LRD_FREEZE_NONE, ws)      # no bias gradient: no column sums
    for k in ("dU", "dV", "db"):
        assert torch.equal(got[k], again[k])
    assert rel_err(dU, got["dU"].double().cpu().numpy()) <= 2 ** -8 and rel_err(dV, got["dV"].double().cpu().numpy()) <= 2 ** -8   # one rounding apart


@pytest.mark.parametrize("n,tokens,stride_rank", [(4, 1000, 96), (3, 300, 192)])
def test_group_of_layers(n, tokens, stride_rank):
    """All gradients of a group whose data chains run in one launch equal each layer's own within one rounding."""
    r, K = stride_rank, 768
    cases = [wl.random_factor_case(tokens, K, K, r, "bf16", 950 + i) for i in range(n)]
    descs = [b.linear_desc(tokens, K, K, r, b.LRD_BF16)] * n
    alone = [run_linear(c, b.LRD_FREEZE_NONE) for c in cases]
    t = {k: [torch.from_numpy(c[k]).to("cuda", torch.bfloat16) for c in cases] for k in ("X", "dY", "V", "U")}
    out = {k: [torch.full_like(a[k], float("nan")) for a in alone] for k in ("dX", "dU", "dV", "db")}
    ws = [torch.empty(b.lrd_linear_workspace_bytes(descs[0], b.LRD_FREEZE_NONE, 1), dtype=torch.uint8, device="cuda") for _ in range(n)]
    b.lrd_linear_group_bwd(descs, t["dY"], t["X"], t["V"], t["U"], [a["Z"] for a in alone], out["dX"], out["dU"], out["dV"], out["db"],
                           b.LRD_FREEZE_NONE, ws)
    assert b.lrd_check_device_status() == b.LRD_OK
    for i in range(n):
        for k in ("dX", "dU", "dV", "db"):
            # dZ is rounded to bf16 after sums in another order: an ulp of some of its values, then one rounding of each result
            assert rel_err(out[k][i], alone[i][k].double().cpu().numpy()) <= 2 ** -7


# freeze mask V: one product (64 wide, pairs, shares through scratch memory, cluster); none: several in one launch
@pytest.mark.parametrize("shape,freeze", [((1021, 1024, 4096, 512), "V"), ((300, 1000, 3528, 1000), "V"), ((5000, 1032, 520, 520), "V"), ((9000, 264, 4096, 264), "V"),
                                          ((4097, 768, 776, 200), "V"), ((130, 264, 328, 64), "U"), ((1000, 520, 1000, 136), "NONE"), ((70, 4096, 4096, 504), "NONE")],
                         ids=lambda x: "x".join(map(str, x)) if isinstance(x, tuple) else x)
def test_adding_to_the_callers_gradients(shape, freeze):
    """The accumulating backward gives exactly the sum of what the buffers held and the plain backward's gradients."""
    M, K, N, r = shape
    f = getattr(b, "LRD_FREEZE_" + freeze)
    g = torch.Generator(device="cuda").manual_seed(M)
    X, dY, V, U, Z = (torch.randn(*s, device="cuda", generator=g).to(torch.bfloat16) for s in ((M, K), (M, N), (K, r), (N, r), (M, r)))
    desc = b.linear_desc(M, K, N, r, b.LRD_BF16)
    ws = torch.empty(b.lrd_linear_workspace_bytes(desc, f, 2), dtype=torch.uint8, device="cuda")
    start = [torch.randn(*s, device="cuda", generator=g).mul_(M ** 0.5).to(torch.bfloat16) for s in ((N, r), (K, r), (N,))]
    plain, summed = [torch.zeros_like(t) for t in start], [t.clone() for t in start]
    dX = torch.empty_like(X)
    x, z = None if freeze == "V" else X, None if freeze == "U" else Z
    b.lrd_linear_bwd(desc, dY, x, V, U, z, dX, *plain, f, ws)
    b.lrd_linear_bwd_accumulate(desc, dY, x, V, U, z, dX, *summed, f, ws)
    assert b.lrd_check_device_status() == b.LRD_OK
    for s, p, q in zip(start, plain, summed):
        assert torch.equal(q, (s.float() + p.float()).to(torch.bfloat16))
