"""Every form that a weight gradient or a split data product can take, asked for by name: tile width x split x products per
launch, plain and adding, with shares of the reduction that are empty, end inside a stage, or are of unequal length.  A call
that cannot run in the form asked for is refused, so what passes here has run in it."""
import pytest
import torch

from paper_2309_03824_b200 import binding as b
from paper_2309_03824_b200 import workloads as wl
from test_gpu_tucker import check_tucker

from helpers import check_linear, run_linear

SINGLE = [(1, c, s) for c in (64, 128, 192) for s in range(1, 9) if c % (8 * s) == 0]
PAIRS = [(2, c, s) for c in (128, 256) for s in (1, 2, 4)]
# tokens, K, N, r: one k-block (all shares but the first empty); shares that end inside a stage of two, ragged rows and columns
SHAPES = [(40, 136, 264, 72), (1100, 200, 136, 104)]


@pytest.fixture
def forms():
    yield
    b.lrd_wgrad_tuning()
    b.lrd_data_split_tuning()


gpu = pytest.mark.gpu


@gpu
@pytest.mark.parametrize("form", SINGLE + PAIRS, ids=lambda f: "x".join(map(str, f)))
def test_one_product(form, forms):
    b.lrd_wgrad_tuning(*form)
    for shape in SHAPES:
        for freeze in (b.LRD_FREEZE_U, b.LRD_FREEZE_V):                # dV; dU with the bias gradient
            case = wl.random_factor_case(*shape, "bf16", 500 + shape[0])
            got, _ = check_linear(case, freeze)
            again = run_linear(case, freeze)
            assert all(torch.equal(got[k], again[k]) for k in ("dU", "dV", "db"))


@gpu
@pytest.mark.parametrize("form", SINGLE + [f for f in PAIRS if f[1] == 256], ids=lambda f: "x".join(map(str, f)))
def test_two_products_in_one_launch(form, forms):
    b.lrd_wgrad_tuning(*form)
    for shape in SHAPES:
        check_linear(wl.random_factor_case(*shape, "bf16", 510 + shape[0]), b.LRD_FREEZE_NONE)
    # reductions of unequal length: dA over the input pixels of a strided convolution, dB over its output pixels
    check_tucker(wl.random_tucker_case(3, 13, 11, 72, 136, 40, 48, 3, "bf16", 520, stride=2), b.LRD_TK_FREEZE_CORE)


@gpu
@pytest.mark.parametrize("form", [f for f in SINGLE if f[2] in (1, 2, 8)] + [(2, 256, 1), (2, 256, 4)], ids=lambda f: "x".join(map(str, f)))
@pytest.mark.parametrize("adding", [False, True])
def test_eight_products_in_one_launch_and_adding(form, adding, forms):
    M, K, N, r, n = 150, 264, 264, 64, 4
    cases = [wl.random_factor_case(M, K, N, r, "bf16", 530 + i) for i in range(n)]
    t = {k: [torch.from_numpy(c[k]).to("cuda", torch.bfloat16) for c in cases] for k in ("X", "dY", "V", "U")}
    descs = [b.linear_desc(M, K, N, r, b.LRD_BF16)] * n
    Z = [(x.float() @ v.float()).to(torch.bfloat16) for x, v in zip(t["X"], t["V"])]
    out = {k: [torch.ones(*s, dtype=torch.bfloat16, device="cuda") for _ in range(n)] for k, s in (("dX", (M, K)), ("dU", (N, r)), ("dV", (K, r)), ("db", (N,)))}
    ws = [torch.empty(b.lrd_linear_workspace_bytes(descs[0], b.LRD_FREEZE_NONE, 2), dtype=torch.uint8, device="cuda") for _ in range(n)]
    b.lrd_wgrad_tuning(*form)
    if adding:                           # (a group has no adding form: its layers one by one, two products a launch)
        for i in range(n):
            b.lrd_linear_bwd_accumulate(descs[i], t["dY"][i], t["X"][i], t["V"][i], t["U"][i], Z[i], *(out[k][i] for k in ("dX", "dU", "dV", "db")),
                                        b.LRD_FREEZE_NONE, ws[i])
    else:
        n0 = b.lrd_launch_count()
        b.lrd_linear_group_bwd(descs, t["dY"], t["X"], t["V"], t["U"], Z, out["dX"], out["dU"], out["dV"], out["db"], b.LRD_FREEZE_NONE, ws)
        assert b.lrd_launch_count() - n0 == 2
    assert b.lrd_check_device_status() == b.LRD_OK
    for i in range(n):
        dY, X = t["dY"][i].double(), t["X"][i].double()
        dZ = (dY @ t["U"][i].double()).to(torch.bfloat16).double()
        for k, ref in (("dU", dY.T @ Z[i].double()), ("dV", X.T @ dZ), ("db", dY.sum(0))):
            # one rounding of the product and, adding, one of the sum; dV is formed from a dZ that may be rounded the other way
            assert float((out[k][i].double() - ref - int(adding)).abs().max() / ref.abs().max()) <= 2 ** -7, k


@gpu
@pytest.mark.parametrize("form", SINGLE, ids=lambda f: "x".join(map(str, f)))
def test_filter_gradient(form, forms):
    b.lrd_wgrad_tuning(*form)
    check_tucker(wl.random_tucker_case(1, 5, 7, 40, 24, 16, 24, 3, "bf16", 540), b.LRD_TK_FREEZE_FACTORS)
    check_tucker(wl.random_tucker_case(4, 15, 13, 88, 96, 72, 40, 3, "bf16", 541, stride=2), b.LRD_TK_FREEZE_FACTORS)


@gpu
@pytest.mark.parametrize("columns", [64, 128])
@pytest.mark.parametrize("split", [2, 4, 8])
def test_split_data_products(columns, split, forms):
    """Both products of a pass, with a bias, more shares than k-blocks, and more tiles than clusters at once."""
    b.lrd_data_split_tuning(columns, split)
    for shape in [(40, 136, 264, 72), (300, 1096, 136, 120), (2500, 264, 1032, 136)]:
        case = wl.random_factor_case(*shape, "bf16", 550 + shape[0])
        for freeze in (b.LRD_FREEZE_NONE, b.LRD_FREEZE_U):
            check_linear(case, freeze, path=b.LRD_PATH_UNFUSED)


@gpu
def test_a_form_that_no_kernel_has_is_refused(forms):
    b.lrd_wgrad_tuning(2, 128, 1)                                      # several products share a launch on pairs 256 wide only
    with pytest.raises(b.LrdError) as e:
        run_linear(wl.random_factor_case(*SHAPES[0], "bf16", 560), b.LRD_FREEZE_NONE)
    assert e.value.status == b.LRD_ERR_UNSUPPORTED


def test_override_values():
    for bad in [(1, 256, 1), (1, 64, 3), (1, 192, 5), (2, 64, 1), (2, 256, 3), (3, 64, 1), (0, 64, 1), (1, 0, 0)]:
        with pytest.raises(b.LrdError):
            b.lrd_wgrad_tuning(*bad)
    for bad in [(192, 2), (64, 3), (64, 0), (0, 2)]:
        with pytest.raises(b.LrdError):
            b.lrd_data_split_tuning(*bad)


@gpu
@pytest.mark.parametrize("form", SINGLE, ids=lambda f: "x".join(map(str, f)))
@pytest.mark.parametrize("shape", SHAPES + [(130, 72, 1000, 8)], ids=lambda s: "x".join(map(str, s)))
def test_adding_leaves_the_rest_alone(form, shape, forms):
    """Gradients added to buffers with a leading dimension of their own: ragged rows and columns, and nothing outside them."""
    M, K, N, r = shape
    case = wl.random_factor_case(M, K, N, r, "bf16", 570 + M)
    X, V, U, dY = (torch.from_numpy(case[k]).to("cuda", torch.bfloat16) for k in ("X", "V", "U", "dY"))
    Z, ld = (X.float() @ V.float()).to(torch.bfloat16), r + 24
    desc = b.linear_desc(M, K, N, r, b.LRD_BF16)
    desc.ldu = ld
    Up, dU = (torch.full((N, ld), 3.0, dtype=torch.bfloat16, device="cuda") for _ in range(2))
    Up[:, :r] = U
    db, dX = torch.ones(N, dtype=torch.bfloat16, device="cuda"), torch.empty_like(X)
    ws = torch.empty(b.lrd_linear_workspace_bytes(desc, b.LRD_FREEZE_V, 2), dtype=torch.uint8, device="cuda")
    b.lrd_wgrad_tuning(*form)
    b.lrd_linear_bwd_accumulate(desc, dY, None, V, Up, Z, dX, dU, None, db, b.LRD_FREEZE_V, ws)
    assert b.lrd_check_device_status() == b.LRD_OK
    ref = dY.double().T @ Z.double()
    # one rounding of the product, one of the sum
    assert float((dU[:, :r].double() - ref - 3).abs().max() / (ref.abs().max() + 3)) <= 2 ** -7
    assert float((db.double() - dY.double().sum(0) - 1).abs().max() / dY.double().sum(0).abs().max()) <= 2 ** -7
    assert bool((dU[:, r:] == 3).all())


SPECIAL = [0x0000, 0x8000, 0x0001, 0x807f, 0x0040, 0x0080, 0x80ff, 0x3f80, 0xbf80, 0x3f81, 0x7b80, 0x7f00, 0x7f7f, 0xff7f, 0x7f80, 0xff80, 0x7fc0]


@gpu
@pytest.mark.parametrize("form", [f for f in SINGLE if f[2] in (1, 3, 8)] + PAIRS[::3], ids=lambda f: "x".join(map(str, f)))
def test_adding_special_values(form, forms):
    """Infinities and their opposites, NaN, sums that overflow, subnormals: the fp32 sum of what stood there and the product, rounded once."""
    M, K, N, r = 64, 136, 264, 64
    S = torch.tensor(SPECIAL, dtype=torch.int32).to(torch.int16).view(torch.bfloat16).cuda()
    dY, Z = torch.zeros(M, N, dtype=torch.bfloat16, device="cuda"), torch.zeros(M, r, dtype=torch.bfloat16, device="cuda")
    dY[0], Z[0] = S.repeat(N // len(S) + 1)[:N], 1                     # dU[n][c] = dY[0][n], whatever c
    V, U = torch.zeros(K, r, dtype=torch.bfloat16, device="cuda"), torch.zeros(N, r, dtype=torch.bfloat16, device="cuda")
    before = S.repeat(r // len(S) + 1)[:r].repeat(N, 1)
    dU, alone = before.clone(), torch.empty(N, r, dtype=torch.bfloat16, device="cuda")
    dX, db = torch.empty(M, K, dtype=torch.bfloat16, device="cuda"), torch.zeros(N, dtype=torch.bfloat16, device="cuda")
    desc = b.linear_desc(M, K, N, r, b.LRD_BF16)
    ws = torch.empty(b.lrd_linear_workspace_bytes(desc, b.LRD_FREEZE_V, 2), dtype=torch.uint8, device="cuda")
    b.lrd_wgrad_tuning(*form)
    b.lrd_linear_bwd_accumulate(desc, dY, None, V, U, Z, dX, dU, None, db, b.LRD_FREEZE_V, ws)
    b.lrd_linear_bwd(desc, dY, None, V, U, Z, dX, alone, None, db, b.LRD_FREEZE_V, ws)
    assert b.lrd_check_device_status() == b.LRD_OK
    want = (alone.float() + before.float()).to(torch.bfloat16)
    assert bool(((dU.view(torch.int16) == want.view(torch.int16)) | (dU.isnan() & want.isnan())).all())
    assert bool(alone[:17].isinf().any()) and bool(want.isnan().any())
