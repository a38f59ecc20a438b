"""Weight gradients on pairs of SMs: both tile widths, one, two and four pairs per tile, shares of the reduction that end inside
a stage, rows and columns that hang over the last tile, and the bias gradient; repeated calls give the same bits."""
import pytest
import torch

from paper_2309_03824_b200 import binding as b
from paper_2309_03824_b200 import workloads as wl

from helpers import check_linear, run_linear

pytestmark = pytest.mark.gpu


# shapes where the estimates choose pairs, when this was written (tile width, pairs): 128 x 1, 256 x 1, 256 x 1, 256 x 2, 256 x 4
# (every form by name: test_gpu_forms.py)
@pytest.mark.parametrize("shape", [(60, 1032, 4096), (300, 3528, 1000), (1021, 4096, 1288), (5000, 264, 4096), (5000, 1032, 520)])
def test_dense_weight_gradient(shape):
    """The undecomposed layer's dW and bias gradient."""
    M, K, N = shape
    g = torch.Generator(device="cuda").manual_seed(M)
    X, dY, W = (torch.randn(*s, device="cuda", generator=g).to(torch.bfloat16) for s in ((M, K), (M, N), (N, K)))
    desc = b.linear_desc(M, K, N, 0, b.LRD_BF16)
    ws = torch.empty(b.lrd_dense_workspace_bytes(desc, 1), dtype=torch.uint8, device="cuda")
    runs = []
    for _ in range(2):
        dX, dW, db = torch.empty_like(X), torch.full_like(W, float("nan")), torch.full((N,), float("nan"), dtype=torch.bfloat16, device="cuda")
        b.lrd_dense_bwd(desc, dY, X, W, dX, dW, db, ws)
        runs.append((dW, db))
    assert b.lrd_check_device_status() == b.LRD_OK
    assert all(torch.equal(p, q) for p, q in zip(*runs))
    for got, ref in zip(runs[0], (dY.double().T @ X.double(), dY.double().sum(0))):
        # fp32 sums of bf16 products, one rounding: 2^-8 of each value, and the sums' own error far below it
        assert float((got.double() - ref).abs().max() / ref.abs().max()) <= 2 ** -8


@pytest.mark.parametrize("shape", [(1030, 4096, 4096, 264), (8192, 1024, 4096, 512)], ids=["one_pair", "two_pairs"])
def test_factor_gradients(shape):
    """dU, dV and the bias gradient of a decomposed layer, beside the data pass and alone."""
    case = wl.random_factor_case(*shape, "bf16", 680 + shape[0])
    got, _ = check_linear(case, b.LRD_FREEZE_NONE)
    again = run_linear(case, b.LRD_FREEZE_NONE)
    for k in ("dU", "dV", "db"):
        assert torch.equal(got[k], again[k])
