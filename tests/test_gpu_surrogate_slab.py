"""conv3 walked along z (few output channels) against the per-plane rows GEMM.

Both kernels sum every output's products in the same order (x-shift, pair of
chunk planes, z-tap, y-tap, 16 channels) on the same tensor-core instruction,
so outputs must agree bit for bit; the rows GEMM itself is compared with the
FP64 oracle in test_gpu_surrogate.py.  Grids cover every box depth (2 to 16
planes), boxes at both ends of the volume, rows of 8 to 64 voxels, more boxes
than SMs and fewer, and each epilogue form (bias and ReLU, fused head, mask and
addend, two destinations)."""
import pytest

pytestmark = pytest.mark.gpu


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


CASES = [  # B, D, H, W, c0, c1, cout; two 128-voxel tiles per z-plane or more (else K-steps of four planes)
    (1, 2, 16, 16, 32, 0, 32), (3, 2, 16, 16, 16, 0, 16), (1, 4, 8, 64, 32, 32, 32),
    (2, 8, 16, 32, 16, 0, 32), (5, 16, 32, 32, 32, 0, 16), (1, 64, 64, 64, 32, 0, 32),
    (1, 8, 32, 8, 64, 0, 16), (2, 16, 8, 32, 32, 0, 64), (9, 16, 16, 16, 32, 0, 32),
]


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


@pytest.mark.parametrize("B,D,H,W,c0,c1,cout", CASES)
def test_forward_equals_rows_gemm(env, B, D, H, W, c0, c1, cout):
    torch, spnn = env
    gen = torch.Generator(device="cuda").manual_seed(B * 1000 + D * 100 + cout)
    x0 = _planes(torch, gen, B, D, H, W, c0)
    x1 = _planes(torch, gen, B, D, H, W, c1) if c1 else None
    w = torch.randn((27, c0 + c1, cout), generator=gen, device="cuda") * 0.1
    bias = torch.randn((cout,), generator=gen, device="cuda")
    hw, hb = torch.randn((cout,), generator=gen, device="cuda"), torch.randn((1,), generator=gen, device="cuda")
    pk = torch.empty(spnn.spnn_packed_elems(spnn.CONV3, c0 + c1, cout), dtype=torch.bfloat16, device="cuda")
    spnn.spnn_pack_weights(spnn.CONV3, c0 + c1, cout, spnn.PACK_FWD, w, pk)

    def run():
        y = spnn.planes_empty(B, D, H, W, cout)
        head = torch.empty((B, D, H, W), dtype=torch.float32, device="cuda")
        spnn.spnn_layer_forward(spnn.CONV3, (B, D, H, W), x0, x1, pk, bias, cout, True, y, hw, hb, head)
        return y, head

    (ya, ha), (yb, hb_) = _both(spnn, run)
    assert torch.equal(ya, yb) and torch.equal(ha, hb_)
    assert float(ya.float().abs().sum()) > 0


@pytest.mark.parametrize("B,D,H,W,c0,c1,cout", [(2, 8, 16, 32, 32, 0, 32), (1, 16, 16, 16, 32, 32, 32),
                                                (3, 4, 32, 32, 16, 0, 64), (4, 16, 32, 64, 16, 0, 32)])
def test_input_gradient_equals_rows_gemm(env, B, D, H, W, c0, c1, cout):
    torch, spnn = env
    gen = torch.Generator(device="cuda").manual_seed(B + D + W)
    dy = _planes(torch, gen, B, D, H, W, cout)
    add, mask = _planes(torch, gen, B, D, H, W, c0), _planes(torch, gen, B, D, H, W, c0)
    w = torch.randn((27, c0 + c1, cout), generator=gen, device="cuda") * 0.1
    pk = torch.empty(spnn.spnn_packed_elems(spnn.CONV3, c0 + c1, cout), dtype=torch.bfloat16, device="cuda")
    spnn.spnn_pack_weights(spnn.CONV3, c0 + c1, cout, spnn.PACK_DGRAD, w, pk)

    def run():
        dx0 = spnn.planes_empty(B, D, H, W, c0)
        dx1 = spnn.planes_empty(B, D, H, W, c1) if c1 else None
        spnn.spnn_layer_dgrad(spnn.CONV3, (B, D, H, W), dy, pk, c0, c1, dx0, addend0=add, mask0=mask, dx1=dx1)
        return (dx0, dx1) if c1 else (dx0,)

    a, b = _both(spnn, run)
    assert all(torch.equal(p, q) for p, q in zip(a, b))
    assert float(a[0].float().abs().sum()) > 0
