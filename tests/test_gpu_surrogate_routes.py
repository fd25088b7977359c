"""Calls of the surrogate's layers that more than one kernel could serve: each of
the kernels by name of its option, and what every one of them refuses."""
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def S():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2604_13929_gb300 import build
    build.build()
    from paper_2604_13929_gb300 import spnn
    yield spnn
    for key, value in (("wgrad_halo", 1), ("conv_planes", 0), ("rows_persistent", 2)):
        spnn.spnn_set_option(key, value)


def planes(gen, c, *grid):
    return torch.randn((c // 8, *grid, 8), generator=gen, device="cuda").to(torch.bfloat16)


@pytest.mark.parametrize("option", [0, 1, 2])
@pytest.mark.parametrize("cout", [272, 320, 512])
def test_wgrad_refuses_more_than_256_output_channels(S, cout, option):
    gen = torch.Generator(device="cuda").manual_seed(cout)
    grid = (1, 4, 8, 16)
    x, dy = planes(gen, 16, *grid), planes(gen, cout, *grid)
    dw = torch.zeros((27, 16, cout), device="cuda")
    S.spnn_set_option("wgrad_halo", option)
    with pytest.raises(S.SpnnError) as e:
        S.spnn_layer_wgrad(S.CONV3, grid, x, None, dy, dw, None)
    assert e.value.code == S.SPNN_EINVAL
    S.spnn_status()
    assert float(dw.abs().sum()) == 0


# layers that the automatic choice gives to the row-window kernel, on the halo kernel: 2 to 10
# planes per CTA, one or two sources, two CTAs per SM on 32-voxel runs (16 + 16 -> 32), walks of
# several slabs, samples and runs per row
HALO = [(2, 4, 8, 32, 32, 0, 32), (2, 4, 8, 32, 32, 32, 32), (2, 4, 8, 32, 16, 0, 32), (2, 4, 8, 32, 48, 0, 32),
        (2, 4, 8, 32, 80, 0, 16), (2, 4, 8, 32, 16, 16, 32), (2, 4, 8, 32, 16, 16, 16), (1, 2, 4, 64, 32, 0, 32),
        (1, 16, 4, 16, 32, 0, 32), (3, 1, 8, 32, 32, 0, 32), (1, 8, 16, 32, 32, 32, 64)]


# the row-window kernel where a CTA takes a single plane of a source, or fewer of one source
# than of the other (the automatic choice)
ROWS = [(1, 4, 8, 16, 8, 8, 16), (2, 4, 4, 32, 8, 8, 32), (1, 4, 4, 32, 8, 8, 64), (1, 4, 8, 8, 8, 40, 32),
        (1, 2, 8, 16, 40, 8, 64), (2, 4, 8, 32, 16, 0, 16)]


@pytest.mark.parametrize("option,B,D,H,W,c0,c1,cout", [(2, *c) for c in HALO] + [(1, *c) for c in ROWS])
def test_conv3_wgrad_against_oracle(S, option, B, D, H, W, c0, c1, cout):
    """The bound of test_gpu_surrogate.py: 2^-12 of the sum of the products' magnitudes."""
    from oracle import unet_oracle as U
    gen = torch.Generator(device="cuda").manual_seed(1000 * B + 100 * D + W + c0 + cout)
    x0, x1 = planes(gen, c0, B, D, H, W), planes(gen, c1, B, D, H, W) if c1 else None
    dy = planes(gen, cout, B, D, H, W)
    voxels = lambda t: S.from_planes(t).double().cpu().numpy()                    # noqa: E731
    x = voxels(x0 if x1 is None else torch.cat([x0, x1]))
    ref, mag = U.conv3_wgrad(x, voxels(dy)), U.conv3_wgrad(abs(x), abs(voxels(dy)))
    dw = torch.zeros((27, c0 + c1, cout), device="cuda")
    db = torch.zeros(cout, device="cuda")
    S.spnn_set_option("wgrad_halo", option)
    S.spnn_layer_wgrad(S.CONV3, (B, D, H, W), x0, x1, dy, dw, db)
    S.spnn_status()
    for got, r, m in zip((dw, db), ref, mag):
        assert (abs(got.double().cpu().numpy() - r) <= 2.0 ** -12 * m + 1e-6).all()


@pytest.mark.parametrize("B,D,H,W,c0,c1,cout", [(2, 8, 16, 32, 16, 16, 32), (5, 16, 32, 32, 32, 0, 32),
                                                (3, 16, 16, 16, 32, 32, 128)])
def test_rows_gemm_conv3_is_independent_of_its_grid(S, B, D, H, W, c0, c1, cout):
    """conv3 on the rows GEMM (two chunk planes per K-step set: not the z-walk), one CTA
    per tile and persistent grids, up to more tiles than CTAs: identical bits."""
    gen = torch.Generator(device="cuda").manual_seed(B + D)
    x0, x1 = planes(gen, c0, B, D, H, W), planes(gen, c1, B, D, H, W) if c1 else None
    w = torch.randn((27, c0 + c1, cout), generator=gen, device="cuda") * 0.1
    bias = torch.randn(cout, generator=gen, device="cuda")
    pk = torch.empty(S.spnn_packed_elems(S.CONV3, c0 + c1, cout), dtype=torch.bfloat16, device="cuda")
    S.spnn_pack_weights(S.CONV3, c0 + c1, cout, S.PACK_FWD, w, pk)
    S.spnn_set_option("conv_planes", 2)
    outs = []
    for grid in (0, 1, 2, 3):
        S.spnn_set_option("rows_persistent", grid)
        y = S.planes_empty(B, D, H, W, cout)
        S.spnn_layer_forward(S.CONV3, (B, D, H, W), x0, x1, pk, bias, cout, True, y)
        S.spnn_status()
        outs.append(y)
    assert all(torch.equal(y, outs[0]) for y in outs[1:]) and float(outs[0].float().abs().sum()) > 0


@pytest.mark.parametrize("B,n,skew", [(1, 16, 0), (64, 16, 0), (3, 24, 0), (1, 32, 0), (5, 32, 1), (700, 8, 3), (2, 64, 5)])
def test_pack_input_porosity(S, B, n, skew):
    """Channel 7 is each sample's pore fraction, counted by one block per sample or several,
    from masks at any byte offset."""
    gen = torch.Generator(device="cuda").manual_seed(n + B)
    flat = torch.zeros(B * n ** 3 + skew, dtype=torch.uint8, device="cuda")
    mask = flat[skew:].view(B, n, n, n)
    level = torch.linspace(0.0, 1.0, B, device="cuda").view(B, 1, 1, 1)
    mask.copy_((torch.rand((B, n, n, n), generator=gen, device="cuda") < level).to(torch.uint8))
    optics = torch.tensor([[0.5, 0.005, 0.7]] * B, device="cuda")
    for _ in range(2):                                   # the second call may find the first one's scratch
        x = S.planes_empty(B, n, n, n, 16)
        S.spnn_pack_input(mask, optics, x)
        phi = S.from_planes(x)[..., 7]
        want = mask.view(B, -1).double().mean(dim=1).to(torch.float32).to(torch.bfloat16)
        assert torch.equal(phi.reshape(B, -1), want[:, None].expand(B, n ** 3))
