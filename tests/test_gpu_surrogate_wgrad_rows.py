"""conv3 weight gradient on row windows against the per-tap kernel.

The two sum the same BF16 products in FP32 in different orders, so they agree
within the accumulation bound of test_gpu_surrogate.py, 2^-12 of the sum of the
products' magnitudes (the per-tap kernel on |x| and |dy|); the per-tap kernel is
compared with the FP64 oracle there.  Cases: runs of 8, 16 and 32 voxels, the
fewest rows of each, 1 to 4 planes per CTA with ragged last splits, two sources,
several blocks of output channels, single z-planes, and a weight gradient that is
not 16-byte aligned."""
import pytest

pytestmark = pytest.mark.gpu

CASES = [  # B, D, H, W, c0, c1, cout, offset of dw in floats
    (1, 2, 4, 32, 16, 0, 32, 0), (2, 1, 8, 16, 32, 0, 16, 0), (1, 8, 8, 8, 32, 0, 32, 0),
    (3, 4, 8, 8, 80, 0, 64, 0), (1, 16, 2, 32, 48, 0, 64, 0), (2, 4, 4, 16, 64, 64, 64, 0),
    (1, 4, 16, 64, 16, 48, 32, 0), (1, 8, 8, 16, 128, 0, 128, 0), (2, 8, 8, 8, 64, 0, 256, 0),
    (1, 8, 16, 32, 32, 32, 32, 1), (1, 64, 64, 64, 32, 0, 32, 0),
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
    spnn.spnn_set_option("wgrad_halo", 1)


@pytest.mark.parametrize("B,D,H,W,c0,c1,cout,off", CASES)
def test_row_windows_equal_per_tap_kernel(env, B, D, H, W, c0, c1, cout, off):
    torch, spnn = env
    gen = torch.Generator(device="cuda").manual_seed(D * 100 + W + c0 + cout)

    def planes(c):
        return torch.randn((c // 8, B, D, H, W, 8), generator=gen, device="cuda").to(torch.bfloat16)

    x0, x1, dy = planes(c0), planes(c1) if c1 else None, planes(cout)

    def run(option, f, bias=True):
        spnn.spnn_set_option("wgrad_halo", option)
        n = 27 * (c0 + c1) * cout
        dw = torch.zeros(n + off, device="cuda")[off:]
        db = torch.zeros(cout, device="cuda") if bias else None
        spnn.spnn_layer_wgrad(spnn.CONV3, (B, D, H, W), f(x0), f(x1) if c1 else None, f(dy), dw, db)
        spnn.spnn_status()
        return dw.double(), db.double() if bias else None

    same = lambda t: t                                   # noqa: E731
    dw, db = run(1, same)
    ref_w, ref_b = run(0, same)
    abs_w, abs_b = run(0, torch.abs)
    assert bool(((dw - ref_w).abs() <= 2.0 ** -12 * abs_w + 1e-6).all())
    assert bool(((db - ref_b).abs() <= 2.0 ** -12 * abs_b + 1e-6).all())
    no_bias, _ = run(1, same, bias=False)
    assert bool(((no_bias - ref_w).abs() <= 2.0 ** -12 * abs_w + 1e-6).all())
