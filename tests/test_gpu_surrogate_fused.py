"""The fused kernels of the surrogate's training step against the separate
calls they stand for: data bit for bit (the same FP32 operations in the same
order), sums over the pixels to FP32 rounding (their order differs: at most
log2(n) + 64 roundings of partial sums, so 1e-5 of the sum of magnitudes)."""
import ctypes

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def env():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1812_00118_gb300 import build, lbm as L
    build.build()
    return torch, L.load(), torch.cuda.current_stream().cuda_stream


def p(t, off=0):
    return ctypes.c_void_p(t.data_ptr() + off * t.element_size()) if t is not None else None


def rnd(torch, *shape, seed=0, dtype=None):
    g = torch.Generator(device="cuda").manual_seed(seed)
    v = torch.randn(*shape, generator=g, device="cuda")
    return v if dtype is None else v.to(dtype)


@pytest.mark.parametrize("N,H,W,ci,co,csy", [(1, 4, 128, 32, 32, 64), (2, 8, 24, 64, 128, 128), (1, 3, 256, 16, 32, 36),
                                             (1, 16, 16, 256, 64, 64), (2, 6, 64, 32, 16, 24)])
def test_conv_relu(env, N, H, W, ci, co, csy):
    torch, lib, s = env
    M, b16 = N * H * W, torch.bfloat16
    x, w, b = rnd(torch, M, ci, dtype=b16), rnd(torch, co, 9, ci, seed=1, dtype=b16), rnd(torch, co, seed=2)
    a, y, z = torch.zeros(M, co, device="cuda"), torch.zeros(M, csy, device="cuda", dtype=b16), None
    z = torch.zeros_like(y)
    assert lib.lbm_sg_conv3x3(p(x), ci, p(w), p(b), p(a), co, N, H, W, ci, co, s) == 0
    assert lib.lbm_sg_relu(p(a), co, p(y), csy, M, co, s) == 0
    assert lib.lbm_sg_conv3x3_relu(p(x), ci, p(w), p(b), p(z), csy, N, H, W, ci, co, s) == 0
    assert torch.equal(y, z) and lib.lbm_sg_status(s) == 0


@pytest.mark.parametrize("mode", ["direct", "up", "pooled"])
@pytest.mark.parametrize("N,H,W,C,cs", [(1, 2, 2, 4, 4), (2, 6, 10, 12, 20), (1, 64, 96, 32, 64), (3, 16, 34, 128, 256)])
def test_relu_grad(env, mode, N, H, W, C, cs):
    torch, lib, s = env
    M, b16 = N * H * W, torch.bfloat16
    act = rnd(torch, M, cs, dtype=b16).relu()
    up = 2 if mode == "up" else 1
    g, gp = rnd(torch, M * up * up, cs, seed=1), rnd(torch, M // 4, cs, seed=2) if mode == "pooled" else None
    t, q = torch.zeros(M, C, device="cuda"), torch.zeros(M, C, device="cuda")
    if mode == "up":
        assert lib.lbm_sg_upsample_bwd(p(g), cs, p(t), C, N, 2 * H, 2 * W, C, 2, s) == 0
    elif mode == "pooled":
        assert lib.lbm_sg_pool_bwd(p(gp), cs, p(q), C, N, H, W, C, 2, s) == 0
        assert lib.lbm_sg_add(p(g), cs, p(q), C, p(t), C, M, C, s) == 0
    else:
        t.copy_(g[:, :C])
    v, v16, w16 = torch.zeros(M, C, device="cuda"), *(torch.zeros(M, C, device="cuda", dtype=b16) for _ in range(2))
    pre = act.float().contiguous()
    assert lib.lbm_sg_relu_bwd(p(t), C, p(pre), cs, p(v), p(v16), M, C, s) == 0
    gb, scr = torch.zeros(C, device="cuda"), torch.zeros(64 * C, device="cuda")
    assert lib.lbm_sg_relu_grad(p(g), cs, up, p(gp), cs if gp is not None else 0, p(act), cs, p(w16), p(gb), p(scr),
                                scr.numel(), N, H, W, C, s) == 0
    assert torch.equal(v16, w16)
    err = (gb.double() - v.double().sum(0)).abs()
    assert (err <= 1e-5 * v.double().abs().sum(0) + 1e-30).all()


def test_relu_grad_refuses(env):
    torch, lib, s = env
    g, a = torch.zeros(64, 8, device="cuda"), torch.zeros(64, 8, device="cuda", dtype=torch.bfloat16)
    o, gb, scr = torch.zeros_like(a), torch.zeros(8, device="cuda"), torch.zeros(4096, device="cuda")
    ok = [p(g), 8, 1, None, 0, p(a), 8, p(o), p(gb), p(scr), 4096, 1, 8, 8, 8, s]
    assert lib.lbm_sg_relu_grad(*ok) == 0
    for k, bad in ((0, None), (0, p(g, 1)), (1, 6), (2, 3), (5, p(a, 1)), (6, 4), (10, 7), (14, 6), (3, p(g))):
        args = list(ok)
        args[k] = bad
        assert lib.lbm_sg_relu_grad(*args) == -1, k


@pytest.mark.parametrize("n", [1, 255, 8192, 8192 * 40 + 7])
def test_mse_grad(env, n):
    torch, lib, s = env
    x, t, d = rnd(torch, n, 4), rnd(torch, n, 4, seed=1), rnd(torch, n, 16, seed=2)
    g, g16, h16 = torch.zeros(n, 16, device="cuda"), *(torch.ones(n, 16, device="cuda", dtype=torch.bfloat16) for _ in (0, 1))
    f64 = lambda k: torch.zeros(k, dtype=torch.float64, device="cuda")
    la, lb, scr, gb = f64(1), f64(1), f64(2 * 512), torch.ones(16, device="cuda")
    assert lib.lbm_sg_mse(p(x), 4, p(d), 16, p(t), 4, p(g), p(scr), p(la), n, 4, s) == 0
    assert lib.lbm_sg_to_bf16(p(g), 16, p(g16), 16, n, 16, s) == 0
    g4 = torch.zeros(n, 4, device="cuda")
    assert lib.lbm_sg_mse_grad(p(x), p(d), p(t), p(h16), p(g4), p(gb), p(scr), p(lb), n, s) == 0
    assert torch.equal(g16, h16) and torch.equal(g4, g[:, :4])
    assert lb.item() == pytest.approx(la.item(), rel=1e-13)
    odd = torch.empty(4 * n + 1, device="cuda")[1:].view(n, 4)   # a target on any address
    odd.copy_(t)
    k16, lc = torch.ones_like(h16), f64(1)
    assert lib.lbm_sg_mse_grad(p(x), p(d), p(odd), p(k16), p(g4), p(gb), p(scr), p(lc), n, s) == 0
    assert torch.equal(k16, h16) and lc.item() == lb.item()
    err = (gb.double() - g.double().sum(0)).abs()
    assert (err <= 1e-5 * g.double().abs().sum(0)).all() and (gb[4:] == 0).all()


@pytest.mark.parametrize("N,H,W,C,cs", [(2, 4, 6, 8, 8), (1, 66, 34, 32, 64), (3, 8, 2, 128, 136)])
def test_wide_pool_and_upsample(env, N, H, W, C, cs):
    """16-byte groups against the per-element kernels (reached by an odd offset)."""
    torch, lib, s = env
    b16 = torch.bfloat16
    buf = rnd(torch, N * H * W * cs + 8, dtype=b16)
    odd = torch.empty(buf.numel() + 1, dtype=b16, device="cuda")[1:]
    odd.copy_(buf)
    for name, rows in (("lbm_sg_pool", N * H * W // 4), ("lbm_sg_upsample", N * H * W)):
        y, z = (torch.zeros(rows * cs, dtype=b16, device="cuda") for _ in range(2))
        fn = getattr(lib, name)
        assert fn(p(buf), cs, p(y), cs, N, H, W, C, 2, s) == 0
        assert fn(p(odd), cs, p(z), cs, N, H, W, C, 2, s) == 0
        assert torch.equal(y, z)


def test_adam_layers(env):
    torch, lib, s = env
    from paper_1812_00118_gb300 import lbm as L
    shapes = [(16, 32), (64, 16), (128, 128)]
    arr, refs, keep = (L.lbm_sg_layer * len(shapes))(), [], []
    for k, (ci, co) in enumerate(shapes):
        t = dict(w=rnd(torch, co, 9, ci, seed=k), mw=rnd(torch, co, 9, ci, seed=k + 10), vw=rnd(torch, co, 9, ci, seed=k + 20).abs(),
                 gw=rnd(torch, co, 9, ci, seed=k + 30), b=rnd(torch, co, seed=k + 40), mb=rnd(torch, co, seed=k + 50),
                 vb=rnd(torch, co, seed=k + 60).abs(), gb=rnd(torch, co, seed=k + 70),
                 w16=torch.zeros(co, 9, ci, dtype=torch.bfloat16, device="cuda"),
                 wt=torch.zeros(ci, 9, co, dtype=torch.bfloat16, device="cuda"))
        keep.append(t)
        r = {n: v.clone() for n, v in t.items()}
        assert lib.lbm_sg_adam(p(r["w"]), p(r["mw"]), p(r["vw"]), p(r["gw"]), r["w"].numel(), 1e-3, 0.9, 0.999, 1e-8, 3,
                               p(r["w16"]), s) == 0
        assert lib.lbm_sg_adam(p(r["b"]), p(r["mb"]), p(r["vb"]), p(r["gb"]), co, 1e-3, 0.9, 0.999, 1e-8, 3, None, s) == 0
        assert lib.lbm_sg_weight_flip(p(r["w16"]), p(r["wt"]), ci, co, s) == 0
        refs.append(r)
        for n, v in t.items():
            setattr(arr[k], n, v.data_ptr())
        arr[k].ci, arr[k].co = ci, co
    assert lib.lbm_sg_adam_layers(arr, len(shapes), 1e-3, 0.9, 0.999, 1e-8, 3, s) == 0
    for t, r in zip(keep, refs):
        for n in t:
            assert torch.allclose(t[n].float(), r[n].float(), rtol=1e-6 if n not in ("w16", "wt") else 8e-3, atol=1e-9), n


def conv_reference(torch, x, w, b, N, H, W):
    """Periodic 3x3 convolution in float64: x (M, ci), w (co, 9, ci)."""
    img = x.double().view(N, H, W, -1)
    out = b.double().view(1, 1, 1, -1).expand(N, H, W, -1)
    for t in range(9):
        out = out + torch.roll(img, (1 - t // 3, 1 - t % 3), (1, 2)) @ w[:, t].double().T
    return out.reshape(N * H * W, -1)


@pytest.mark.parametrize("N,H,W,ci,co", [
    (1, 2, 8, 16, 16), (2, 4, 8, 32, 128), (3, 33, 16, 64, 32), (1, 8, 250, 32, 48), (2, 7, 40, 128, 64),   # flat tiles
    (2, 64, 64, 256, 64), (1, 64, 64, 64, 128), (3, 32, 32, 128, 128), (1, 16, 62, 64, 128), (1, 1, 16, 16, 16), (1, 32, 32, 128, 128), (1, 16, 16, 32, 96),
    (1, 1, 128, 16, 16), (1, 2, 128, 128, 32), (1, 3, 128, 64, 128), (2, 9, 256, 32, 16), (1, 200, 128, 16, 32),   # march
    (1, 16, 64, 256, 128), (1, 4, 128, 256, 64)])                                                        # tap kernel
def test_conv_paths_exact_on_integers(env, N, H, W, ci, co):
    """Every path of the convolution and of the weight gradient on integers
    small enough that every sum is exact: equal to float64 bit for bit."""
    torch, lib, s = env
    g = torch.Generator(device="cuda").manual_seed(N + H * W + ci * co)
    r = lambda lo, hi, *sh: torch.randint(lo, hi + 1, sh, generator=g, device="cuda").bfloat16()
    M = N * H * W
    x, w, gy, b = r(-2, 2, M, ci), r(-2, 2, co, 9, ci), r(-1, 1, M, co), r(-5, 5, co).float()
    y, gw = torch.full((M, co), 7.0, device="cuda"), torch.zeros(co, 9, ci, device="cuda")
    assert lib.lbm_sg_conv3x3(p(x), ci, p(w), p(b), p(y), co, N, H, W, ci, co, s) == 0
    assert torch.equal(y.double(), conv_reference(torch, x, w, b, N, H, W))
    n = lib.lbm_sg_wgrad_scratch_floats(N, H, W, ci, co)
    scr = torch.full((n,), float("nan"), device="cuda")
    assert lib.lbm_sg_conv3x3_wgrad(p(x), ci, p(gy), co, p(gw), p(scr), n, N, H, W, ci, co, s) == 0
    img, gi = x.double().view(N, H, W, ci), gy.double().view(N * H * W, co)
    want = torch.stack([gi.T @ torch.roll(img, (1 - t // 3, 1 - t % 3), (1, 2)).reshape(-1, ci) for t in range(9)], 1)
    assert torch.equal(gw.double(), want) and lib.lbm_sg_status(s) == 0


@pytest.mark.parametrize("npix", [1, 255, 257, 4095, 16 * 1000, 16383, 16384, 65537])
@pytest.mark.parametrize("C", [4, 12, 16, 20, 128])
def test_bias_sums_one_order(env, npix, C):
    """The bias sums are the same bits on every path: rows in 16-byte groups, one
    channel per block (reached by an address off a 16-byte boundary), and inside
    lbm_sg_relu_grad and lbm_sg_mse_grad."""
    torch, lib, s = env
    g = rnd(torch, npix, C, seed=3)
    odd = torch.empty(npix * C + 1, device="cuda")[1:].view(npix, C)
    odd.copy_(g)
    act = torch.ones(npix, C, device="cuda", dtype=torch.bfloat16)
    a, b, c = (torch.zeros(C, device="cuda") for _ in range(3))
    scr, ga = torch.zeros(64 * C, device="cuda"), torch.zeros_like(act)
    assert lib.lbm_sg_bias_grad(p(g), C, p(a), p(scr), npix, C, s) == 0
    assert lib.lbm_sg_bias_grad(p(odd), C, p(b), p(scr), npix, C, s) == 0
    assert lib.lbm_sg_relu_grad(p(g), C, 1, None, 0, p(act), C, p(ga), p(c), p(scr), scr.numel(), 1, 1, npix, C, s) == 0
    assert torch.equal(a, b) and torch.equal(a, c)
    if C == 4:
        x, t, d = rnd(torch, npix, 4), rnd(torch, npix, 4, seed=1), rnd(torch, npix, 16, seed=2)
        g4, g16 = torch.zeros(npix, 4, device="cuda"), torch.zeros(npix, 16, device="cuda", dtype=torch.bfloat16)
        e, want = torch.ones(16, device="cuda"), torch.zeros(4, device="cuda")
        part, loss = (torch.zeros(k, dtype=torch.float64, device="cuda") for k in (1024, 1))
        assert lib.lbm_sg_mse_grad(p(x), p(d), p(t), p(g16), p(g4), p(e), p(part), p(loss), npix, s) == 0
        assert lib.lbm_sg_bias_grad(p(g4), 4, p(want), p(scr), npix, 4, s) == 0
        assert torch.equal(e[:4], want) and (e[4:] == 0).all()
