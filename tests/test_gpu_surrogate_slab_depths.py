"""conv3 walked along z at every box depth, each CTA walking more boxes than it has
accumulator buffers, against the per-plane rows GEMM (same bits, see
test_gpu_surrogate_slab.py).  test_launch_rules.py checks on the CPU that the cases
reach every (output channels, depth) pair on 152 SMs with at least three boxes on
some CTAs, so that a buffer is waited for and used again."""
import pytest

pytestmark = pytest.mark.gpu

# B, D, H, W, input channels, output channels (of the GEMM: its N), box depth
CASES = [
    (39, 4, 16, 32, 32, 16, 2), (40, 8, 16, 32, 16, 16, 4), (6, 32, 32, 64, 32, 16, 8), (12, 32, 32, 64, 16, 16, 16),
    (40, 2, 32, 32, 64, 32, 2), (39, 4, 32, 32, 32, 32, 4), (2, 64, 64, 64, 32, 32, 4), (4, 64, 64, 64, 16, 32, 8),
    (39, 8, 8, 32, 32, 64, 2), (6, 16, 32, 64, 32, 64, 4), (1, 64, 64, 64, 16, 16, 16), (2, 64, 64, 64, 32, 16, 16),
    (64, 8, 16, 32, 32, 32, 8), (80, 16, 16, 8, 16, 32, 4),
]


@pytest.fixture(scope="module")
def env():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2604_13929_gb300 import build
    build.build()
    from paper_2604_13929_gb300 import spnn
    yield torch, spnn
    spnn.spnn_set_option("conv_planes", 0)


def _planes(torch, gen, B, D, H, W, c):
    return torch.randn((c // 8, B, D, H, W, 8), generator=gen, device="cuda").to(torch.bfloat16)


def _both(spnn, run):
    """Outputs of the z-walk and of the rows GEMM (two chunk planes per K-step)."""
    out = []
    for planes in (0, 2):
        spnn.spnn_set_option("conv_planes", planes)
        out.append(run())
        spnn.spnn_status()
    return out


@pytest.mark.parametrize("B,D,H,W,cin,cout,depth", CASES)
def test_forward(env, B, D, H, W, cin, cout, depth):
    torch, spnn = env
    gen = torch.Generator(device="cuda").manual_seed(B * 1000 + D * 100 + cout)
    x = _planes(torch, gen, B, D, H, W, cin)
    w = torch.randn((27, cin, cout), generator=gen, device="cuda") * 0.1
    bias = torch.randn((cout,), generator=gen, device="cuda")
    pk = torch.empty(spnn.spnn_packed_elems(spnn.CONV3, cin, cout), dtype=torch.bfloat16, device="cuda")
    spnn.spnn_pack_weights(spnn.CONV3, cin, cout, spnn.PACK_FWD, w, pk)

    def run():
        y = spnn.planes_empty(B, D, H, W, cout)
        spnn.spnn_layer_forward(spnn.CONV3, (B, D, H, W), x, None, pk, bias, cout, True, y)
        return y

    a, b = _both(spnn, run)
    assert torch.equal(a, b) and float(a[:, -1, -1].float().abs().sum()) > 0


@pytest.mark.parametrize("B,D,H,W,cin,cout,depth", CASES)
def test_input_gradient(env, B, D, H, W, cin, cout, depth):
    """N of this GEMM is the layer's input channels: a layer cout -> cin in the table's terms."""
    torch, spnn = env
    gen = torch.Generator(device="cuda").manual_seed(B + D + W + cout)
    dy = _planes(torch, gen, B, D, H, W, cin)
    mask = _planes(torch, gen, B, D, H, W, cout)
    w = torch.randn((27, cout, cin), generator=gen, device="cuda") * 0.1
    pk = torch.empty(spnn.spnn_packed_elems(spnn.CONV3, cout, cin), dtype=torch.bfloat16, device="cuda")
    spnn.spnn_pack_weights(spnn.CONV3, cout, cin, spnn.PACK_DGRAD, w, pk)

    def run():
        dx = spnn.planes_empty(B, D, H, W, cout)
        spnn.spnn_layer_dgrad(spnn.CONV3, (B, D, H, W), dy, pk, cout, 0, dx, mask0=mask)
        return dx

    a, b = _both(spnn, run)
    assert torch.equal(a, b) and float(a[:, -1, -1].float().abs().sum()) > 0
