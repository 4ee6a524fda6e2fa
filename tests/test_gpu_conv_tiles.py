"""The tensor-core convolution over its tilings, channel layouts, output
slices and masks, against a 64-bit convolution (needs a GPU)."""
import pytest

pytestmark = pytest.mark.gpu


def conv64(x, w):
    """3x3 convolution, zero padding, NHWC, float64; w [N, 3, 3, C]."""
    import torch
    B, H, W, C = x.shape
    p = torch.zeros(B, H + 2, W + 2, C, dtype=torch.float64, device=x.device)
    p[:, 1:-1, 1:-1] = x
    y = torch.zeros(B, H, W, w.shape[0], dtype=torch.float64, device=x.device)
    for ky in range(3):
        for kx in range(3):
            y += p[:, ky:ky + H, kx:kx + W] @ w[:, ky, kx].T
    return y


# images of whole tiles, one row or column around a tile's edge, stacked images
# whose tiles span two of them, narrow images as one row, single pixels
@pytest.mark.parametrize("B,H,W", [(1, 16, 8), (2, 17, 33), (3, 15, 7), (5, 20, 50), (7, 10, 25), (4, 5, 30),
                                   (9, 3, 31), (3, 1, 1), (2, 1, 64), (2, 64, 1), (70, 16, 40)])
# one to many channel planes of every width (the last two: a tap's channels at a
# time); channel blocks of odd sizes
@pytest.mark.parametrize("cin,cout", [(8, 32), (16, 2), (32, 96), (48, 24), (64, 10), (96, 40), (192, 64),
                                      (128, 264), (512, 48), (768, 256), (1024, 24)])
def test_conv_tilings(B, H, W, cin, cout):
    import torch
    from paper_2509_01827_gb300 import build, surrogate
    build.build()
    L = surrogate.sg()
    dev = "cuda"
    g = torch.Generator(device=dev).manual_seed(B * 1000 + cin)
    P, ld, off = B * H * W, cin + 8, 8
    xw = torch.randn(P, ld, device=dev, generator=g).bfloat16()
    x = xw[:, off:]  # a channel slice of a wider tensor
    w = (torch.randn(cout, 3, 3, cin, device=dev, generator=g) / (3 * cin ** 0.5)).bfloat16()
    b = torch.randn(cout, device=dev, generator=g)
    mk = torch.randn(P, cout, device=dev, generator=g).bfloat16()
    st = torch.cuda.current_stream().cuda_stream
    t0 = surrogate.timeouts()
    x64, w64 = x.double().view(B, H, W, cin), w.double()
    ref = conv64(x64, w64).view(P, cout)
    # rounding to BF16 (2^-9 relative) and of the FP32 sums (9 cin terms, each
    # at most 2^-22 of the sum of magnitudes off, truncation included)
    tol = 2.0 ** -8 * ref.abs() + 9 * cin * 2.0 ** -22 * conv64(x64.abs(), w64.abs()).view(P, cout) + 1e-30
    for pad, bias, relu, mask in ((0, b, 1, None), (6, None, 0, mk), (16, b, 0, mk)):
        y = torch.full((P, cout + 2 * pad), 7.0, device=dev).bfloat16()
        rc = L.cem_sg_conv3x3(x.data_ptr(), B, H, W, cin, ld, w.data_ptr(),
                              None if bias is None else bias.data_ptr(), cout, relu,
                              None if mask is None else mask.data_ptr(), cout, y.data_ptr(),
                              cout + 2 * pad, pad, st)
        assert rc == 0
        want = ref + (0 if bias is None else bias.double())
        if relu:
            want = want.clamp(min=0)
        if mask is not None:
            want = torch.where(mask.double() > 0, want, torch.zeros_like(want))
        got = y[:, pad:pad + cout].double()
        slack = tol + 2.0 ** -8 * (0 if bias is None else bias.double().abs())
        assert bool(((got - want).abs() <= slack).all()), float((got - want).abs().max())
        # nothing beside the slice is written
        assert bool((y[:, :pad] == 7).all()) and bool((y[:, pad + cout:] == 7).all())
    assert surrogate.timeouts() == t0


# the same tilings for the weight gradient; 64 x 9 x 31 and 5 x 160 x 100 take several
# tile ranges and workspace slots, 2 x 64 x 640 several flushes of a range
@pytest.mark.parametrize("B,H,W", [(1, 16, 8), (2, 17, 33), (5, 20, 50), (7, 10, 25), (9, 3, 31), (3, 1, 1),
                                   (2, 1, 64), (64, 9, 31), (5, 160, 100), (2, 64, 640)])
@pytest.mark.parametrize("cin,cout", [(32, 32), (96, 32), (32, 64), (64, 64), (192, 96), (64, 128), (128, 256),
                                      (512, 64), (24, 40), (8, 32), (8, 96)])
@pytest.mark.parametrize("with_bias", [True, False])
def test_wgrad_tilings(B, H, W, cin, cout, with_bias):
    import torch
    from paper_2509_01827_gb300 import build, surrogate
    build.build()
    L = surrogate.sg()
    dev = "cuda"
    g = torch.Generator(device=dev).manual_seed(B * 1000 + cin)
    P, ld = B * H * W, cin + 16
    x = torch.randn(P, ld, device=dev, generator=g).bfloat16()[:, 8:8 + cin]  # a channel slice
    dy = torch.randn(P, cout, device=dev, generator=g).bfloat16()
    need = L.cem_sg_wgrad_workspace(B, H, W, cin, cout)
    ws = torch.full((need + 64,), 0xff, dtype=torch.uint8, device=dev)  # NaNs, and a guard behind
    dw = torch.full((cout, 3, 3, cin), float("nan"), device=dev)
    db = torch.full((cout,), float("nan"), device=dev)
    t0 = surrogate.timeouts()
    rc = L.cem_sg_conv3x3_wgrad(x.data_ptr(), ld, dy.data_ptr(), cout, B, H, W, cin, cout, dw.data_ptr(),
                                db.data_ptr() if with_bias else None, ws.data_ptr(), need,
                                torch.cuda.current_stream().cuda_stream)
    assert rc == 0 and surrogate.timeouts() == t0
    assert bool((ws[need:] == 0xff).all())
    x64, y64 = x.double().view(B, H, W, cin), dy.double().view(B, H, W, cout)
    p = torch.zeros(B, H + 2, W + 2, cin, dtype=torch.float64, device=dev)
    p[:, 1:-1, 1:-1] = x64
    yf = y64.reshape(P, cout)
    for ky in range(3):
        for kx in range(3):
            w = p[:, ky:ky + H, kx:kx + W].reshape(P, cin)
            # FP32 sums of at most 8192 pixels in steps of 16, each step at most 2^-23
            # of the magnitudes off
            tol = 512 * 2.0 ** -23 * (yf.abs().T @ w.abs()) + 1e-30
            assert bool(((dw[:, ky, kx].double() - yf.T @ w).abs() <= tol).all()), (ky, kx)
    if with_bias:
        tol = 512 * 2.0 ** -23 * yf.abs().sum(0) + 1e-30
        assert bool(((db.double() - yf.sum(0)).abs() <= tol).all())
    else:
        assert bool(torch.isnan(db).all())


# the head's row accesses (8, 16 and 32 channels, others, an odd pixel count) and the
# pooling and upsampling kernels' row walk against plain sums
@pytest.mark.parametrize("C", [8, 12, 16, 24, 32])
@pytest.mark.parametrize("P", [1, 4095, 4097, 70001])
def test_head_rows(C, P):
    import torch
    from paper_2509_01827_gb300 import build, surrogate
    build.build()
    L, st = surrogate.sg(), torch.cuda.current_stream().cuda_stream
    g = torch.Generator(device="cuda").manual_seed(C)
    x = torch.randn(P, C, device="cuda", generator=g).bfloat16()
    w, dz = (torch.randn(n, device="cuda", generator=g) for n in (C, P))
    b = torch.randn(1, device="cuda", generator=g)
    z, dx = torch.empty(P, device="cuda"), torch.empty_like(x)
    dw, db = torch.empty(C, device="cuda"), torch.empty(1, device="cuda")
    nb = L.cem_sg_head_workspace(P, C)
    ws = torch.empty(nb, dtype=torch.uint8, device="cuda")
    assert L.cem_sg_head_fwd(x.data_ptr(), P, C, w.data_ptr(), b.data_ptr(), z.data_ptr(), st) == 0
    assert L.cem_sg_head_bwd(x.data_ptr(), P, C, w.data_ptr(), dz.data_ptr(), dx.data_ptr(), dw.data_ptr(),
                             db.data_ptr(), ws.data_ptr(), nb, st) == 0
    x64, w64, d64 = x.double(), w.double(), dz.double()
    mag = (x64.abs() @ w64.abs()) + b.double().abs()
    assert bool(((z.double() - (x64 @ w64 + b.double())).abs() <= (C + 1) * 2.0 ** -23 * mag).all())
    want = torch.where(x > 0, dz[:, None] * w[None], torch.zeros((), device="cuda")).bfloat16()
    assert torch.equal(dx, want)
    # at most 64 values a thread, 32 lanes, 8 warps and P / 4096 chunks in FP32
    n = (64 + 32 + 8 + P // 4096 + 8) * 2.0 ** -24
    assert bool(((dw.double() - d64 @ x64).abs() <= 4 * n * (d64.abs() @ x64.abs())).all())
    assert float((db.double() - d64.sum()).abs()) <= 4 * n * 8 * float(d64.abs().sum())
