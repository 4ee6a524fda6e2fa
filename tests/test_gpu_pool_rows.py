"""Pooling, upsampling and their gradients on images of any width, against
plain sums; and narrow images take about the time of wide ones with as many pixels
(needs a GPU)."""
import pytest

pytestmark = pytest.mark.gpu


def _ops(B, H, W, C, g):
    """The four operations on images of H x W (2H x 2W) pixels: calls, and their results' buffers."""
    import torch
    from paper_2509_01827_gb300 import surrogate
    L, st = surrogate.sg(), torch.cuda.current_stream().cuda_stream
    rnd = lambda *s: torch.randn(*s, device="cuda", generator=g).bfloat16()
    ld, off = 2 * C + 8, C + 8  # the skip and the upsampled channels are slices of wider tensors
    x, small, wide = rnd(B, 2 * H, 2 * W, C), rnd(B, H, W, C), rnd(B, 2 * H, 2 * W, ld)
    y, dx, up, dsm = torch.empty_like(small), torch.empty_like(x), torch.full_like(wide, 7.0), torch.empty_like(small)
    p = lambda t: t.data_ptr()
    calls = [lambda: L.cem_sg_maxpool2(p(x), C, B, H, W, C, p(y), st),
             lambda: L.cem_sg_maxpool2_bwd(p(x), C, p(small), p(wide), ld, off, B, H, W, C, 1, p(dx), st),
             lambda: L.cem_sg_upsample2(p(small), B, H, W, C, p(up), ld, off, st),
             lambda: L.cem_sg_upsample2_bwd(p(wide), ld, B, H, W, C, p(small), C, p(dsm), st)]
    return calls, x, small, wide, y, dx, up, dsm, off


@pytest.mark.parametrize("B,H,W,C", [(1, 1, 1, 8), (3, 5, 1, 8), (2, 7, 3, 24), (5, 4, 31, 8), (2, 3, 32, 64),
                                     (1, 6, 33, 64), (2, 1, 257, 8), (700, 2, 2, 16)])
def test_pool_and_upsample(B, H, W, C):
    import torch
    from paper_2509_01827_gb300 import build
    build.build()
    calls, x, small, wide, y, dx, up, dsm, off = _ops(B, H, W, C, torch.Generator(device="cuda").manual_seed(W))
    assert [f() for f in calls] == [0, 0, 0, 0]
    win = lambda t: t.view(B, H, 2, W, 2, -1).permute(0, 1, 3, 5, 2, 4).reshape(B, H, W, -1, 4)
    back = lambda t: t.view(B, H, W, -1, 2, 2).permute(0, 1, 4, 2, 5, 3).reshape(B, 2 * H, 2 * W, -1)
    v, sk = win(x).float(), win(wide[..., off:off + C].contiguous()).float()
    m = v.amax(-1)
    assert torch.equal(y.float(), m)
    eq = v == m[..., None]
    first = eq & (eq.int().cumsum(-1) == 1)
    want = torch.where(first, small.float()[..., None], torch.zeros(())) + sk
    want = torch.where(v > 0, want, torch.zeros(()))
    assert torch.equal(dx, back(want).bfloat16())
    want = torch.full_like(wide, 7.0)
    want[..., off:off + C] = small.repeat_interleave(2, 1).repeat_interleave(2, 2)
    assert torch.equal(up, want)
    q = win(wide[..., :C].contiguous()).float()
    want = ((q[..., 0] + q[..., 1]) + q[..., 2]) + q[..., 3]
    want = torch.where(small.float() > 0, want, torch.zeros(()))
    assert torch.equal(dsm, want.bfloat16())


def test_narrow_images_take_no_longer():
    import torch
    from paper_2509_01827_gb300 import build
    build.build()
    t = []
    for B, H, W in ((4096, 4, 4), (1, 16, 4096)):  # as many pixels
        g = torch.Generator(device="cuda").manual_seed(1)
        t.append([])
        state = _ops(B, H, W, 8, g)
        for f in state[0]:
            best = 1e9
            for _ in range(8):
                a, b = torch.cuda.Event(True), torch.cuda.Event(True)
                a.record()
                for _ in range(20):
                    f()
                b.record()
                b.synchronize()
                best = min(best, a.elapsed_time(b))
            t[-1].append(best)
    # a block to an image row took 4 to 15 times as long
    assert all(n < 2.5 * w for n, w in zip(*t)), t
