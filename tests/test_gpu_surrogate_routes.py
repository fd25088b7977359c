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
