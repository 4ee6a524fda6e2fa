"""Weight gradients of inputs that hold infinities and NaN at the images' borders:
an entry is non-finite only where its sum has a non-finite term, whichever tiles
the kernels take (needs a GPU)."""
import pytest

pytestmark = pytest.mark.gpu


# ragged and exact whole tiles, stacked images, narrow images as one row, the gathering
# kernel; one workspace slot (few tiles) and many
@pytest.mark.parametrize("B,H,W", [(1, 16, 8), (2, 17, 33), (7, 10, 25), (5, 20, 50), (1, 1, 3), (40, 33, 40)])
@pytest.mark.parametrize("cin,cout", [(8, 32), (32, 64), (64, 64), (192, 96), (512, 64), (24, 40)])
@pytest.mark.parametrize("every", [False, True])
def test_nonfinite_borders(B, H, W, cin, cout, every):
    import torch
    from paper_2509_01827_gb300 import build, surrogate
    build.build()
    L = surrogate.sg()
    g = torch.Generator(device="cuda").manual_seed(B * 1000 + cin)
    P = B * H * W
    x = torch.randn(B, H, W, cin, device="cuda", generator=g).bfloat16()
    dy = torch.randn(B, H, W, cout, device="cuda", generator=g).bfloat16()
    inf, nan = float("inf"), float("nan")
    if every:
        x[:] = nan
    else:
        x[0, 0, W // 2, 0] = inf         # top
        x[B - 1, H - 1, 0, 1] = -inf     # lower left corner
        x[B // 2, H // 2, W - 1, 2] = nan  # right
        x[0, 0, :, 3] = inf              # the whole top row
        x[B - 1, H // 2, W // 2, 4] = inf  # inside
        dy[0, H - 1, W - 1, 6] = inf     # and one of the other operand
    need = L.cem_sg_wgrad_workspace(B, H, W, cin, cout)
    ws = torch.empty(need, dtype=torch.uint8, device="cuda")
    dw = torch.empty(cout, 3, 3, cin, device="cuda")
    db = torch.empty(cout, device="cuda")
    rc = L.cem_sg_conv3x3_wgrad(x.data_ptr(), cin, dy.data_ptr(), cout, B, H, W, cin, cout, dw.data_ptr(),
                                db.data_ptr(), ws.data_ptr(), need, torch.cuda.current_stream().cuda_stream)
    assert rc == 0
    p = torch.zeros(B, H + 2, W + 2, cin, dtype=torch.float64, device="cuda")
    p[:, 1:-1, 1:-1] = x.double()
    yf = dy.double().reshape(P, cout)
    for ky in range(3):
        for kx in range(3):
            w = p[:, ky:ky + H, kx:kx + W].reshape(P, cin)
            # no product of a zero with an infinity is left to a matrix multiplication's order
            want = torch.stack([(yf[:, o:o + 1] * w).sum(0) for o in range(0, cout, 3)])
            got = dw[::3, ky, kx].double()
            assert torch.equal(torch.isnan(got), torch.isnan(want)), (ky, kx)
            inf_w = torch.isinf(want)
            assert torch.equal(got[inf_w], want[inf_w]) and torch.equal(torch.isinf(got), inf_w), (ky, kx)
            ok = torch.isfinite(want)
            f = torch.nan_to_num(w, 0, 0, 0).abs()
            mag = (torch.nan_to_num(yf, 0, 0, 0).abs().T @ f)[::3]
            # FP32 sums of at most 8192 pixels in steps of 16, each step at most 2^-23 of the magnitudes off
            assert bool(((got - want).abs()[ok] <= (512 * 2.0 ** -23 * mag + 1e-30)[ok]).all()), (ky, kx)
