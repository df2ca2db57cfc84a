"""Performance cases: the calls a user of this library makes, over the range
of sizes, storage types and boundaries they make them on.

    listed()             the named cases
    draw(rng)            one more case of the same ranges
    prepare(case, seed)  fields, simulation, batch or network on the GPU
    run(state)           one pass through the public entry points
    work(case)           bytes and floating-point operations of one pass
    exact(case, seed)    the same results in 64 bits, in plain torch

A case is a dict; "kind" selects what runs:

  sim      lbm.Simulation: `steps` time steps, then the fields of the state
           (lbm_macro) or its checkpoint (lbm_get_populations)
  batch    lbm.Batch: the same for many D2Q9 grids at once
  train    surrogate.Surrogate.train_step of the warm-start U-Net
  warm     warmstart.predict_into: a state jumped ahead by the network
  conv     one convolution layer of the U-Net, forward and backward

The library hands fields out as doubles; a program that keeps snapshots keeps
them in the precision of the stored populations, so run() rounds FP32 results
to float32 and 16-bit ones (scaled like the stored values) to float16.
"""
import ctypes
import math

import numpy as np
import torch

from paper_1812_00118_gb300 import lbm as L
from paper_1812_00118_gb300 import surrogate as SG
from paper_1812_00118_gb300 import warmstart as WS

STORES = {"f64": L.F64, "f32": L.F32, "f16s": L.F16S}
BYTES = {"f64": 8, "f32": 4, "f16s": 2}
OUT = {"f64": torch.float64, "f32": torch.float32, "f16s": torch.float16}
G_SCALE = 1e3          # scale of the stored g of the 16-bit cases


def listed():
    return [
        # Section 4.1 static droplet, the FP64 configuration: a relaxation run
        # advances 100 steps between two looks at the state; the smallest
        # domain, where a step is a launch and little else.  The state is kept
        # as a checkpoint.
        dict(name="drop2d_64_f64", kind="sim", flow="drop", nx=64, ny=64, nz=1, store="f64", steps=100,
             out="checkpoint"),
        # One grid of the time-to-tolerance comparison: some tens of steps, then
        # the fields the convergence check reads.
        dict(name="relax2d_256_f32", kind="sim", flow="drop", nx=256, ny=256, nz=1, store="f32", steps=40,
             out="fields"),
        # Rayleigh-Taylor of Section 4 on its 150 x 600 domain: walls, gravity,
        # a width that is no multiple of a warp.
        dict(name="taylor2d_150x600_f32", kind="sim", flow="taylor", nx=150, ny=600, nz=1, store="f32", steps=40,
             out="fields"),
        # Layered two-phase channel of Section 3: a thin D3Q19 domain between
        # walls, tens of thousands of steps of little work each.
        dict(name="channel3d_4x256x4_f32", kind="sim", flow="channel", nx=4, ny=256, nz=4, store="f32", steps=40,
             out="fields"),
        # The 128^3 static bubble, the library's headline workload.
        dict(name="bubble3d_128_f32", kind="sim", flow="bubble", nx=128, ny=128, nz=128, store="f32", steps=20,
             out="fields"),
        # A static bubble in a box with no round size, run to a checkpoint.
        dict(name="bubble3d_odd_f32", kind="sim", flow="bubble", nx=117, ny=75, nz=90, store="f32", steps=20,
             out="checkpoint"),
        # A bubble carried by a flow with a pressure wave, in 16-bit shifted
        # storage, with the total of phi re-imposed as that needs.
        dict(name="carried3d_128_f16s", kind="sim", flow="carried", nx=128, ny=128, nz=128, store="f16s", steps=10,
             out="fields"),
        # The rising bubble at its specified size: the largest domain, walls at
        # the z ends, gravity.
        dict(name="rising3d_256x256x512_f32", kind="sim", flow="rising", nx=256, ny=256, nz=512, store="f32",
             steps=10, out="fields"),
        # 512 uneven D2Q9 drops and bubbles in one batch, stepped by a graph
        # between two looks at every grid.
        dict(name="batch2d_512_f32", kind="batch", grids=512, lo=32, hi=512, store="f32", steps=20),
        # A training step of the warm-start U-Net on its mini-batch.
        dict(name="train_8x256", kind="train", n=8, h=256, w=256),
        # The warm start of one 256^2 case: four applications of the network
        # and the rebuilt state.
        dict(name="warm_256", kind="warm", size=256, apply=4),
        # The widest full-resolution layer of the U-Net (d1), forward and
        # backward.
        dict(name="conv_8x256_64to32", kind="conv", n=8, h=256, w=256, ci=64, co=32),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choices(["sim2d", "sim3d", "batch", "train", "warm", "conv"], [4, 4, 1, 1, 1, 2])[0]
    if kind == "sim2d":
        flow = rng.choice(["drop", "drop", "taylor"])
        store = rng.choice(["f32", "f32", "f64"])
        top = 400 if store == "f64" else 1000
        return dict(kind="sim", flow=flow, nx=_log(rng, 32, top), ny=_log(rng, 48, top), nz=1, store=store, steps=40,
                    out=rng.choice(["fields", "checkpoint"]))
    if kind == "sim3d":
        flow = rng.choice(["bubble", "drop", "rising", "channel"])
        if flow == "channel":
            return dict(kind="sim", flow=flow, nx=rng.randint(3, 16), ny=_log(rng, 32, 400), nz=rng.randint(3, 16),
                        store=rng.choice(["f32", "f64"]), steps=40, out="fields")
        store = rng.choice(["f32", "f32", "f16s", "f64"])
        if store == "f16s":
            flow = "carried"
        side = {"f64": 72, "f32": 240, "f16s": 240}[store]
        return dict(kind="sim", flow=flow, nx=_log(rng, 24, side), ny=_log(rng, 24, side), nz=_log(rng, 32, side),
                    store=store, steps=10, out="fields" if store == "f16s" else rng.choice(["fields", "checkpoint"]))
    if kind == "batch":
        lo = rng.choice([32, 48, 64])
        return dict(kind="batch", grids=_log(rng, 6, 400), lo=lo, hi=rng.randint(lo + 16, 512), store="f32", steps=20)
    if kind == "train":
        return dict(kind="train", n=rng.randint(1, 8), h=32 * rng.randint(1, 8), w=32 * rng.randint(1, 8))
    if kind == "warm":
        return dict(kind="warm", size=32 * rng.randint(2, 8), apply=rng.randint(1, 4))
    return dict(kind="conv", n=rng.randint(1, 8), h=4 * rng.randint(4, 64), w=4 * rng.randint(4, 64),
                ci=rng.choice([16, 32, 64, 128]), co=rng.choice([16, 32, 64, 128]))


# ---------------------------------------------------------------- flows
def _dev():
    return "cuda" if torch.cuda.is_available() else "cpu"


def _coords(nx, ny, nz):
    r = lambda n: torch.arange(n, dtype=torch.float64, device=_dev())
    return r(nx).view(1, 1, nx), r(ny).view(1, ny, 1), r(nz).view(nz, 1, 1)


def _ball(nx, ny, nz, centre, R, W, drop, wall_z=False):
    """tanh profile of a drop or bubble, periodic distances (z: not across walls)."""
    r2 = 0.0
    for x, n, c, wall in zip(_coords(nx, ny, nz), (nx, ny, nz), centre, (False, False, wall_z)):
        if n > 1:
            d = x - c
            r2 = r2 + (d if wall else torch.remainder(d + n / 2.0, n) - n / 2.0) ** 2
    d = R - torch.sqrt(r2)
    return (0.5 + 0.5 * torch.tanh((2.0 if drop else -2.0) * d / W)).expand(nz, ny, nx).contiguous()


def _flow(case, seed):
    """(parameters, boundaries, force on rho - mean, phi, u, P) of a sim case:
    the set-ups of the tests and the benchmark, with radius, position and
    amplitude from the seed.  phi (nz, ny, nx), u (dim, nz, ny, nx)."""
    rng = np.random.default_rng([seed, 1812])
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    two_d = nz == 1 and case["flow"] in ("drop", "taylor")
    dim = 2 if two_d else 3
    shape = (nz, ny, nx)
    bc = [L.PERIODIC] * 3
    off = rng.uniform(-0.45, 0.45, 3)
    grow = 1.0 + rng.uniform(-0.08, 0.08)
    u = torch.zeros((dim,) + shape, dtype=torch.float64, device=_dev())
    P = torch.zeros(shape, dtype=torch.float64, device=_dev())
    centre = [n / 2 + o for n, o in zip((nx, ny, nz), off)]
    small = min(nx, ny) if two_d else min(nx, ny, nz)
    p = dict(g=(0.0, 0.0, 0.0), force_mode=0)
    if case["flow"] == "drop":
        p.update(M=0.1, W=4.0, sigma=0.01, rho_L=1e-3, rho_H=1.0, nu_L=1.0 / 60.0, nu_H=1.0 / 60.0)
        phi = _ball(nx, ny, nz, centre, small / 4.0 * grow, 4.0, True)
    elif case["flow"] == "taylor":
        p.update(M=5.8e-3, W=2.5, sigma=8.6e-4 / 3, rho_L=1.0 / 3, rho_H=1.0, nu_L=5.7e-3, nu_H=1.9e-3,
                 g=(0.0, -1e-5, 0.0), force_mode=1)
        bc[1] = L.WALL
        x, y, _ = _coords(nx, ny, nz)
        y0 = ny / 2 + 0.1 * grow * min(nx, ny) * torch.cos(2 * math.pi * (x + 0.5 + off[0]) / nx)
        phi = (0.5 + 0.5 * torch.tanh(2 * (y - y0) / 2.5)).expand(shape).contiguous()
    elif case["flow"] == "channel":
        p.update(M=0.1, W=2.5, sigma=0.01, rho_L=1e-3, rho_H=1.0, nu_L=1.7, nu_H=0.17, g=(1e-7, 0.0, 0.0))
        bc[1] = L.WALL
        _, y, _ = _coords(nx, ny, nz)
        phi = (0.5 + 0.5 * torch.tanh(2 * (ny / 2 - 0.5 + off[1] - y) / 2.5)).expand(shape).contiguous()
        P += 2e-5 * torch.cos(math.pi * (y + 0.5) / ny)
        u[0] = (4e-3 * grow * (y + 0.5) * (ny - 0.5 - y) / (ny / 2.0) ** 2).expand(shape)
    elif case["flow"] == "bubble":
        p.update(M=0.1, W=5.0, sigma=1e-3, rho_L=1e-3, rho_H=1.0, nu_L=1e-3, nu_H=1e-3)
        phi = _ball(nx, ny, nz, centre, small * 24.0 / 128.0 * grow, 5.0, False)
    elif case["flow"] == "carried":
        p.update(M=0.1, W=4.0, sigma=1e-3, rho_L=0.1, rho_H=1.0, nu_L=0.1, nu_H=0.1)
        phi = _ball(nx, ny, nz, centre, small / 4.0 * grow, 4.0, False)
        for a, v in enumerate(rng.uniform(0.5, 1.0, dim)):
            u[a] = 0.025 * float(v)
        x, y, z = _coords(nx, ny, nz)
        P += 1e-3 * (torch.cos(2 * math.pi * (x / nx + off[0])) * torch.cos(2 * math.pi * (y / ny + off[1]))
                     + torch.cos(2 * math.pi * (z / nz + off[2])))
    else:   # rising
        p.update(M=0.1, W=4.0, sigma=5e-4, rho_L=1e-3, rho_H=1.0, nu_L=0.1, nu_H=0.01, g=(0.0, 0.0, -1e-6),
                 force_mode=1)
        bc[2] = L.WALL
        centre[2] = nz / 8.0 + max(2.0, small / 16.0) + off[2]
        phi = _ball(nx, ny, nz, centre, small / 8.0 * grow, 4.0, False, wall_z=True)
    return p, bc, dim, phi, u, P


def _params(p, store):
    return L.make_params(store=STORES[store], g_scale=G_SCALE if store == "f16s" else 0.0, **p)


# ---------------------------------------------------------------- LB states
def _sim_state(case, seed):
    p, bc, dim, phi, u, P = _flow(case, seed)
    shape = (case["nx"], case["ny"]) if dim == 2 else (case["nx"], case["ny"], case["nz"])
    sim = L.Simulation(L.D2Q9 if dim == 2 else L.D3Q19, shape, _params(p, case["store"]), bc=tuple(bc))
    if case["store"] == "f16s":
        sim.set_phi_correction(case["steps"])
    sim.init_fields(phi.view(-1), u.view(-1), P.view(-1))
    z = lambda n: torch.zeros(n, dtype=torch.float64, device="cuda")
    s = dict(kind="sim", sim=sim, steps=case["steps"], out=case["out"], store=case["store"])
    if case["out"] == "fields":
        s.update(phi=z(sim.N), P=z(sim.N), ru=z(dim * sim.N))
    else:
        s.update(h=z(sim.Q * sim.N), g=z(sim.Q * sim.N))
    return s


def _rounded(store, phi, P, ru):
    """The fields in the precision the populations are stored in."""
    k, t = (G_SCALE if store == "f16s" else 1.0), OUT[store]
    if store == "f64":
        return dict(phi=phi, P=P, rho_u=ru)
    if k == 1.0:
        return dict(phi=phi.to(t), P=P.to(t), rho_u=ru.to(t))
    return dict(phi=phi.to(t), P=(P * k).to(t), rho_u=(ru * k).to(t))


def _run_sim(s):
    sim = s["sim"]
    sim.step(s["steps"])
    if s["out"] == "fields":
        sim.macro(s["phi"], s["P"], s["ru"])
        return _rounded(s["store"], s["phi"], s["P"], s["ru"])
    sim.get_populations(s["h"], s["g"])
    return dict(h=s["h"].to(OUT[s["store"]]), g=s["g"].to(OUT[s["store"]]))


def _batch_cases(case, seed):
    """Static drops and bubbles of uneven size, as the batched configuration draws them."""
    got = []
    # the sizes belong to the case (every seed steps the same amount of work)
    sides = np.random.default_rng([case["grids"], case["lo"], case["hi"]]).integers(case["lo"], case["hi"] + 1,
                                                                                  case["grids"])
    for k, side in enumerate(sides):
        rng = np.random.default_rng([seed, k])
        side = int(side)
        ratio = math.exp(rng.uniform(math.log(10.0), math.log(1000.0)))
        tau = float(rng.uniform(0.51, 0.8))
        got.append(dict(side=side, R=side / 4.0 + rng.uniform(-1.0, 1.0) * side / 16.0, drop=bool(rng.integers(0, 2)),
                        c=rng.uniform(-0.45, 0.45, 2) + side / 2.0,
                        p=dict(M=0.1, W=float(rng.choice([3.0, 4.0, 5.0])), sigma=0.01, rho_L=1.0 / ratio, rho_H=1.0,
                               nu_L=(tau - 0.5) / 3.0, nu_H=(tau - 0.5) / 3.0)))
    return got


def _batch_phi(c):
    return _ball(c["side"], c["side"], 1, (c["c"][0], c["c"][1], 0.0), c["R"], c["p"]["W"], c["drop"]).view(-1)


def _batch_state(case, seed):
    cases = _batch_cases(case, seed)
    batch = L.Batch([(c["side"], c["side"]) for c in cases], [_params(c["p"], case["store"]) for c in cases])
    batch.set_graph(10)
    n = [c["side"] ** 2 for c in cases]
    zeros = torch.zeros(2 * max(n), dtype=torch.float64, device="cuda")
    for k, c in enumerate(cases):
        batch.grid(k).init_fields(_batch_phi(c), zeros[:2 * n[k]], zeros[:n[k]])
    z = lambda m: torch.zeros(m, dtype=torch.float64, device="cuda")
    phi, P, ru = z(sum(n)), z(sum(n)), z(2 * sum(n))
    views = list(zip(phi.split(n), P.split(n), ru.split([2 * m for m in n])))
    return dict(kind="batch", batch=batch, steps=case["steps"], phi=phi, P=P, ru=ru, views=views, store=case["store"])


def _run_batch(s):
    s["batch"].step(s["steps"])
    for k, (phi, P, ru) in enumerate(s["views"]):
        s["batch"].grid(k).macro(phi, P, ru)
    return _rounded(s["store"], s["phi"], s["P"], s["ru"])


# ---------------------------------------------------------------- network states
def _net_params(seed, last):
    """He-normal weights; `last` scales the output layer (near the identity map)."""
    rng = np.random.default_rng([seed, 7])
    out = {}
    for name, ci, co in SG.LAYERS:
        out[name + ".W"] = rng.normal(0.0, math.sqrt(2.0 / (9 * ci)) * (last if name == "out" else 1.0), (co, ci, 3, 3))
        out[name + ".b"] = rng.normal(0.0, 0.02, co)
    return out


def _images(n, h, w, seed):
    """Normalised (phi, rho u, P) of drops in a gentle flow, and the state they go to: (M, 4) float32."""
    rng = np.random.default_rng([seed, 3])
    x, y, _ = _coords(w, h, 1)
    x, y = x.view(1, w), y.view(h, 1)
    ins, outs = [], []
    for _ in range(n):
        c, R = rng.uniform(0.2, 0.8, 2) * (w, h), min(h, w) * rng.uniform(0.15, 0.3)
        k, ph, amp = rng.integers(1, 4, (8, 2)), rng.uniform(0, 2 * math.pi, 8), rng.normal(0, 0.7, 8)
        wave = [amp[j] * torch.cos(2 * math.pi * (k[j, 0] * x / w + k[j, 1] * y / h) + ph[j]) for j in range(8)]
        ball = lambda r: 0.5 + 0.5 * torch.tanh(0.5 * (r - torch.sqrt((x - c[0]) ** 2 + (y - c[1]) ** 2)))
        ins.append(torch.stack([ball(R), wave[0] + wave[1], wave[2] + wave[3], wave[4] + ball(R)], -1))
        outs.append(torch.stack([ball(R + 0.3), wave[0] * 0.7 + wave[5], wave[2] * 0.7 + wave[6], wave[7] + ball(R)], -1))
    pack = lambda v: torch.stack(v).reshape(n * h * w, 4).float().contiguous()
    return pack(ins), pack(outs)


def _train_state(case, seed):
    x, t = _images(case["n"], case["h"], case["w"], seed)
    return dict(kind="train", net=SG.Surrogate(case["n"], case["h"], case["w"], params=_net_params(seed, 0.1)), x=x, t=t)


def _run_train(s):
    loss = s["net"].train_step(s["x"], s["t"], lr=1e-3)
    return dict(loss=loss, **{name: {k: ly[k] for k in ("gW", "gb", "W", "b")} for name, ly in s["net"].layers.items()})


def _warm_case(case):
    return dict(kind="sim", flow="drop", nx=case["size"], ny=case["size"], nz=1, store="f32")


def _warm_state(case, seed):
    n = case["size"]
    p, bc, dim, phi, u, P = _flow(_warm_case(case), seed)
    prm = _params(p, "f32")
    net = SG.Surrogate(1, n, n, params=_net_params(seed, 0.05))
    sim = L.Simulation(L.D2Q9, (n, n), prm)
    z = lambda m: torch.zeros(m, dtype=torch.float64, device="cuda")
    return dict(kind="warm", net=net, sim=sim, prm=prm, phi0=phi.view(-1).cpu().numpy(), apply=case["apply"],
                phi=z(n * n), P=z(n * n), ru=z(2 * n * n))


def _run_warm(s):
    WS.predict_into(torch, s["net"], s["sim"], s["phi0"], s["prm"], s["apply"])
    s["sim"].macro(s["phi"], s["P"], s["ru"])
    return _rounded("f32", s["phi"], s["P"], s["ru"])


def _conv_inputs(case, seed):
    """bf16 activations (ReLU outputs), weights and output gradients of a layer, and its FP32 bias and gradient."""
    gen = torch.Generator(device=_dev()).manual_seed(seed)
    M, ci, co = case["n"] * case["h"] * case["w"], case["ci"], case["co"]
    r = lambda *sh: torch.randn(*sh, generator=gen, device=_dev())
    g = r(M, co) * (r(M, co) > 0) * 1e-3
    return dict(x=r(M, ci).relu().bfloat16(), w=(r(co, 9, ci) * math.sqrt(2.0 / (9 * ci))).bfloat16(), b=0.05 * r(co),
                g=g, g16=g.bfloat16())


def _conv_state(case, seed):
    s = _conv_inputs(case, seed)
    M, ci, co = case["n"] * case["h"] * case["w"], case["ci"], case["co"]
    z = lambda *sh: torch.zeros(*sh, device="cuda")
    dims = (case["n"], case["h"], case["w"])
    need = L.load().lbm_sg_wgrad_scratch_floats(*dims, ci, co)
    s.update(kind="conv", dims=dims, ci=ci, co=co, M=M, wt=torch.zeros(ci, 9, co, dtype=torch.bfloat16, device="cuda"),
             y=z(M, co), gx=z(M, ci), gw=z(co, 9, ci), gb=z(co), scratch=z(max(int(need), 64 * co)))
    return s


def _run_conv(s):
    lib, st = L.load(), torch.cuda.current_stream().cuda_stream
    p = lambda t: ctypes.c_void_p(t.data_ptr())
    ci, co, dims = s["ci"], s["co"], s["dims"]
    rc = [lib.lbm_sg_conv3x3(p(s["x"]), ci, p(s["w"]), p(s["b"]), p(s["y"]), co, *dims, ci, co, st),
          lib.lbm_sg_conv3x3_wgrad(p(s["x"]), ci, p(s["g16"]), co, p(s["gw"]), p(s["scratch"]), s["scratch"].numel(),
                                   *dims, ci, co, st),
          lib.lbm_sg_bias_grad(p(s["g"]), co, p(s["gb"]), p(s["scratch"]), s["M"], co, st),
          lib.lbm_sg_weight_flip(p(s["w"]), p(s["wt"]), ci, co, st),
          lib.lbm_sg_conv3x3(p(s["g16"]), co, p(s["wt"]), None, p(s["gx"]), ci, *dims, co, ci, st)]
    if any(rc):
        raise RuntimeError("convolution layer: status %s" % rc)
    return dict(y=s["y"], gx=s["gx"], gw=s["gw"], gb=s["gb"])


_PREPARE = dict(sim=_sim_state, batch=_batch_state, train=_train_state, warm=_warm_state, conv=_conv_state)
_RUN = dict(sim=_run_sim, batch=_run_batch, train=_run_train, warm=_run_warm, conv=_run_conv)


def prepare(case, seed):
    return _PREPARE[case["kind"]](case, seed)


def run(state):
    return _RUN[state["kind"]](state)


# ---------------------------------------------------------------- work
def _net_work(n, h, w):
    """Multiply-add FLOPs of one forward pass, and the number of parameters."""
    level = dict(e1=0, e2=1, e3=2, b=3, d3=2, d2=1, d1=0, out=0)
    flops = sum(2.0 * n * (h >> level[k]) * (w >> level[k]) * 9 * ci * co for k, ci, co in SG.LAYERS)
    return flops, sum(9 * ci * co + co for _, ci, co in SG.LAYERS)


def work(case):
    if case["kind"] in ("sim", "batch"):
        # a step reads and writes every population of both sets once; the
        # fields (or the checkpoint) are written once, as doubles
        two_d = case["kind"] == "batch" or case["flow"] in ("drop", "taylor")
        Q, per_lu = (9, 330.0) if two_d else (19, 700.0)
        n = sum(c["side"] ** 2 for c in _batch_cases(case, 0)) if case["kind"] == "batch" \
            else case["nx"] * case["ny"] * case["nz"]
        out = 2 * Q if case.get("out") == "checkpoint" else (4 if two_d else 5)
        return dict(bytes=float(n) * (4 * Q * BYTES[case["store"]] * case["steps"] + 8 * out),
                    flops=float(n) * per_lu * case["steps"])
    if case["kind"] == "train":
        f, k = _net_work(case["n"], case["h"], case["w"])
        m = case["n"] * case["h"] * case["w"]
        # input and target once; parameters and both moments read and written, gradients written
        return dict(bytes=32.0 * m + 28.0 * k, flops=3.0 * f)
    if case["kind"] == "warm":
        f, k = _net_work(1, case["size"], case["size"])
        m = case["size"] ** 2
        return dict(bytes=8.0 * m + 2.0 * k + 72.0 * m + 32.0 * m, flops=f * case["apply"])
    m, ci, co = float(case["n"] * case["h"] * case["w"]), case["ci"], case["co"]
    return dict(bytes=m * (2 * ci + 4 * co + 2 * co + 4 * co + 4 * ci) + 8.0 * 9 * ci * co, flops=3 * 2 * m * 9 * ci * co)


# ---------------------------------------------------------------- 64-bit results
# Velocities in the order the library reports (lbm_lattice_info), user axes.
_C2 = [(0, 0, 0), (1, 0, 0), (-1, 0, 0), (0, 1, 0), (1, 1, 0), (-1, 1, 0), (0, -1, 0), (1, -1, 0), (-1, -1, 0)]
_C3 = [(0, 0, 0), (1, 0, 0), (-1, 0, 0), (0, 1, 0), (1, 1, 0), (-1, 1, 0), (0, -1, 0), (1, -1, 0), (-1, -1, 0),
       (0, 0, 1), (1, 0, 1), (-1, 0, 1), (0, 0, -1), (1, 0, -1), (-1, 0, -1), (0, 1, 1), (0, -1, -1), (0, 1, -1),
       (0, -1, 1)]
_T = 1.0 / 3.0


def _weight(c, three_d):
    k = sum(v * v for v in c)
    return ((1 / 3, 1 / 18, 1 / 36) if three_d else (4 / 9, 1 / 9, 1 / 36))[k]


class _Model:
    """The model of the paper on flat 64-bit fields of one or more grids, whose
    parameters are numbers or one value per node."""

    def __init__(self, grids, three_d):
        """grids: (nx, ny, nz, walls per axis) of each grid, one after the other."""
        self.c = _C3 if three_d else _C2
        self.w = [_weight(c, three_d) for c in self.c]
        self.Q, self.dim = len(self.c), 3 if three_d else 2
        self.opp = [self.c.index(tuple(-v for v in c)) for c in self.c]
        self.N = sum(nx * ny * nz for nx, ny, nz, _ in grids)
        self.near = [None] + [torch.empty(self.N, dtype=torch.int32, device=_dev()) for _ in self.c[1:]]
        self.pull = [None] + [torch.empty(self.N, dtype=torch.int32, device=_dev()) for _ in self.c[1:]]
        at = 0
        for nx, ny, nz, walls in grids:
            i = lambda n: torch.arange(n, device=_dev())
            xyz = (i(nx).view(1, 1, nx), i(ny).view(1, ny, 1), i(nz).view(nz, 1, 1))
            n = nx * ny * nz
            own = torch.arange(at, at + n, device=_dev()).view(nz, ny, nx)
            for k in range(1, self.Q):
                near, src, hit = [], [], torch.zeros(1, 1, 1, dtype=torch.bool, device=_dev())
                for x, m, c, wall in zip(xyz, (nx, ny, nz), self.c[k], walls):
                    near.append((x + c).clamp(0, m - 1) if wall else (x + c) % m)
                    src.append((x - c).clamp(0, m - 1) if wall else (x - c) % m)
                    if wall:
                        hit = hit | (x - c < 0) | (x - c >= m)
                flat = lambda v: at + v[0] + nx * (v[1] + ny * v[2])
                self.near[k][at:at + n] = flat(near).expand(nz, ny, nx).reshape(-1).int()
                p = torch.where(hit, self.opp[k] * self.N + own, k * self.N + flat(src))
                self.pull[k][at:at + n] = p.expand(nz, ny, nx).reshape(-1).int()
            at += n

    def set(self, p, rho_bar=0.0):
        tau = lambda nu: nu / _T + 0.5
        self.p, self.rho_bar, self.rd = p, rho_bar, p["rho_H"] - p["rho_L"]
        self.omL, self.omH = 1.0 / tau(p["nu_L"]), 1.0 / tau(p["nu_H"])
        self.g = p.get("g", (0.0, 0.0, 0.0))

    def _stencil(self, f):
        grad, lap = [torch.zeros_like(f) for _ in range(self.dim)], torch.zeros_like(f)
        for k in range(1, self.Q):
            v = f.index_select(0, self.near[k])
            for a in range(self.dim):
                if self.c[k][a]:
                    grad[a].add_(v, alpha=3.0 * self.c[k][a] * self.w[k])
            lap.add_(v.sub_(f), alpha=6.0 * self.w[k])
        return grad, lap

    def _local(self, phi):
        s, p = {}, self.p
        s["phi"] = phi
        s["grad"], s["lap"] = self._stencil(phi)
        s["rho"] = p["rho_L"] + phi * self.rd
        s["mu"] = 48.0 * p["sigma"] / p["W"] * phi * (phi - 1) * (phi - 0.5) - 1.5 * p["sigma"] * p["W"] * s["lap"]
        fr = s["rho"] - self.rho_bar if p.get("force_mode", 0) == 1 else s["rho"]
        s["F"] = [fr * self.g[a] if self.g[a] else None for a in range(self.dim)]
        return s

    def _dot(self, c, v):
        out = 0.0
        for a in range(self.dim):
            if c[a] and v[a] is not None:
                out = out + (v[a] if c[a] > 0 else -v[a])
        return out

    def _inner(self, u, v):
        out = 0.0
        for a, b in zip(u, v):
            if b is not None:
                out = out + a * b
        return out

    def _flow(self, s, g):
        rho_e = s["rho"] + 0.25 * self.rd * s["lap"]
        s["u"] = []
        for a in range(self.dim):
            m = 0.5 * s["mu"] * s["grad"][a]
            if s["F"][a] is not None:
                m = m + 0.5 * s["F"][a]
            for k in range(1, self.Q):
                if self.c[k][a]:
                    m.add_(g[k], alpha=float(self.c[k][a]))
            s["u"].append(m.div_(rho_e))
        s["P"] = _T * g.sum(0) + 0.5 * _T * self.rd * self._inner(s["u"], s["grad"])

    def _equilibria(self, s):
        """Yields (k, h^eq, K, g^eq) of every direction."""
        p, w, rd = self.p, self.w, self.rd
        u, phi, mu = s["u"], s["phi"], s["mu"]
        usq, ug, uF = self._inner(u, u), self._inner(u, s["grad"]), self._inner(u, s["F"])
        inv = 1.0 / (torch.sqrt(self._inner(s["grad"], s["grad"])) + 1e-10)
        theta = p["M"] / _T / p["W"] * (1.0 - 4.0 * (phi - 0.5) ** 2) * inv
        for k, c in enumerate(self.c):
            cu = self._dot(c, u)
            d = w[k] * (3.0 * cu + 4.5 * cu * cu - 1.5 * usq)        # Gamma - w
            G = d + w[k]
            K = (d * rd + 3.0 * G * mu) * (self._dot(c, s["grad"]) - ug) + 3.0 * G * (self._dot(c, s["F"]) - uF)
            geq = s["rho"] * d + 3.0 * w[k] * s["P"] - 0.5 * K + 0.75 * w[k] * rd * cu * s["lap"]
            heq = phi * G + theta * (w[k] * self._dot(c, s["grad"]))
            yield k, heq, K, geq

    def init(self, phi, u, P):
        s = self._local(phi)
        s["u"], s["P"] = u, P
        h = torch.empty(self.Q, self.N, dtype=torch.float64, device=phi.device)
        g = torch.empty_like(h)
        for k, heq, _, geq in self._equilibria(s):
            h[k], g[k] = heq, geq
        return h, g

    def step(self, h, g, h2, g2):
        """One step of (h, g); the work buffers h2, g2 receive it."""
        s = self._local(h.sum(0))
        self._flow(s, g)
        c, w, D = self.c, self.w, self.dim
        Pi = [[torch.zeros_like(s["phi"]) if b >= a else None for b in range(D)] for a in range(D)]
        it = 1.0 / (self.p["M"] / _T + 0.5)
        for k, heq, K, geq in self._equilibria(s):
            h2[k] = h[k] + (heq - h[k]) * it
            g2[k] = geq + K
            d = g[k] - geq
            for a in range(D):
                for b in range(a, D):
                    if c[k][a] * c[k][b]:
                        Pi[a][b].add_(d, alpha=float(c[k][a] * c[k][b]))
        tr = sum(Pi[a][a] for a in range(D))
        pc = s["phi"].clamp(0.0, 1.0)
        f = 4.5 * (1.0 - (self.omL + pc * (self.omH - self.omL)))
        for k in range(self.Q):
            cc = -_T * tr
            for a in range(D):
                for b in range(a, D):
                    m = c[k][a] * c[k][b] * (1 if a == b else 2)
                    if m:
                        cc = cc + m * Pi[a][b]
            g2[k] += w[k] * f * cc
        del s, Pi
        for src, dst in ((h2, h), (g2, g)):
            dst[0] = src[0]
            for k in range(1, self.Q):
                torch.index_select(src.view(-1), 0, self.pull[k], out=dst[k])

    def fields(self, h, g):
        s = self._local(h.sum(0))
        self._flow(s, g)
        return s["phi"], s["P"], torch.cat([s["rho"] * v for v in s["u"]])


def _exact_fields(store, phi, P, ru):
    k = G_SCALE if store == "f16s" else 1.0
    return dict(phi=phi, P=P * k, rho_u=ru * k)


def _exact_sim(case, seed):
    p, bc, dim, phi, u, P = _flow(case, seed)
    m = _Model([(case["nx"], case["ny"], case["nz"], [b == L.WALL for b in bc])], dim == 3)
    m.set(p, p["rho_L"] + (p["rho_H"] - p["rho_L"]) * float(phi.mean()))
    h, g = m.init(phi.view(-1), [v.reshape(-1) for v in u], P.view(-1))
    h2, g2 = torch.empty_like(h), torch.empty_like(g)
    for _ in range(case["steps"]):
        m.step(h, g, h2, g2)
    if case["out"] == "checkpoint":
        return dict(h=h.view(-1), g=g.view(-1))
    return _exact_fields(case["store"], *m.fields(h, g))


def _exact_batch(case, seed):
    cases = _batch_cases(case, seed)
    m = _Model([(c["side"], c["side"], 1, (False, False, False)) for c in cases], False)
    n = torch.tensor([c["side"] ** 2 for c in cases], device=_dev())
    per_node = lambda key: torch.tensor([c["p"][key] for c in cases], dtype=torch.float64,
                                        device=_dev()).repeat_interleave(n)
    p = dict(M=0.1, sigma=0.01, rho_H=1.0, **{key: per_node(key) for key in ("W", "rho_L", "nu_L")})
    p["nu_H"] = p["nu_L"]
    m.set(p)
    zero = torch.zeros(m.N, dtype=torch.float64, device=_dev())
    h, g = m.init(torch.cat([_batch_phi(c) for c in cases]), [zero, zero], zero)
    h2, g2 = torch.empty_like(h), torch.empty_like(g)
    for _ in range(case["steps"]):
        m.step(h, g, h2, g2)
    phi, P, ru = m.fields(h, g)
    sizes = n.tolist()   # every grid's vector field on its own, x components first
    ru = torch.cat([torch.cat(v) for v in zip(ru[:m.N].split(sizes), ru[m.N:].split(sizes))])
    return _exact_fields(case["store"], phi, P, ru)


def _conv64(x, w, b):
    """Periodic 3x3 convolution of (n, ci, h, w) by (co, ci, 3, 3), one matrix product per tap."""
    out = 0.0
    for dy in range(3):
        for dx in range(3):
            xs = torch.roll(x, (1 - dy, 1 - dx), (2, 3))
            out = out + torch.einsum("nihw,oi->nohw", xs, w[:, :, dy, dx])
    return out if b is None else out + b.view(1, -1, 1, 1)


def _net64(P, x):
    pool = lambda v: torch.nn.functional.avg_pool2d(v, 2)
    up = lambda v: v.repeat_interleave(2, 2).repeat_interleave(2, 3)
    layer = lambda name, v: torch.relu(_conv64(v, P[name + ".W"], P[name + ".b"]))
    s1 = layer("e1", x)
    s2 = layer("e2", pool(s1))
    s3 = layer("e3", pool(s2))
    t3 = layer("d3", torch.cat([s3, up(layer("b", pool(s3)))], 1))
    t2 = layer("d2", torch.cat([s2, up(t3)], 1))
    t1 = layer("d1", torch.cat([s1, up(t2)], 1))
    return _conv64(t1, P["out.W"], P["out.b"])


def _params64(seed, last):
    return {k: torch.tensor(v, dtype=torch.float64, device=_dev()) for k, v in _net_params(seed, last).items()}


def _exact_train(case, seed):
    n, h, w = case["n"], case["h"], case["w"]
    x, t = (v.double().view(n, h, w, 4).permute(0, 3, 1, 2) for v in _images(n, h, w, seed))
    P = {k: v.requires_grad_(True) for k, v in _params64(seed, 0.1).items()}
    loss = ((x + _net64(P, x) - t) ** 2).mean()
    loss.backward()
    out = dict(loss=loss.detach().view(1))
    for name, ci, co in SG.LAYERS:
        cip, cop = (ci + 15) // 16 * 16, (co + 15) // 16 * 16
        W, gW = torch.zeros(2, cop, 9, cip, dtype=torch.float64, device=_dev())
        b, gb = torch.zeros(2, cop, dtype=torch.float64, device=_dev())
        for dst, src in ((W, P[name + ".W"].detach()), (gW, P[name + ".W"].grad)):
            dst[:co, :, :ci] = src.reshape(co, ci, 9).transpose(1, 2)
        b[:co], gb[:co] = P[name + ".b"].detach(), P[name + ".b"].grad
        adam = lambda v, g: v - 1e-3 * g / (g.abs() + 1e-8)      # the first Adam update
        out[name] = dict(gW=gW, gb=gb, W=adam(W, gW), b=adam(b, gb))
    return out


def _exact_warm(case, seed):
    n = case["size"]
    p, _, _, phi0, _, _ = _flow(_warm_case(case), seed)
    P = _params64(seed, 0.05)
    scale = torch.tensor(WS.SCALE, dtype=torch.float64, device=_dev()).view(1, 4, 1, 1)
    x = torch.zeros(1, 4, n, n, dtype=torch.float64, device=_dev())
    x[0, 0] = phi0[0]
    for _ in range(case["apply"]):
        x = x + _net64(P, x)
    phi, rux, ruy, Pr = (x * scale)[0].reshape(4, -1)
    f0 = phi0.view(-1)
    phi = (f0 + 4.0 * f0 * (1.0 - f0) * (phi - f0)).clamp(0.0, 1.0)
    m = 4.0 * phi * (1.0 - phi)
    phi = phi + (f0.sum() - phi.sum()) / m.sum() * m
    return dict(phi=phi, P=Pr, rho_u=torch.cat([rux, ruy]))


def _exact_conv(case, seed):
    s = _conv_inputs(case, seed)
    n, h, w, ci, co = case["n"], case["h"], case["w"], case["ci"], case["co"]
    image = lambda v, c: v.double().view(n, h, w, c).permute(0, 3, 1, 2)
    x = image(s["x"], ci).requires_grad_(True)
    W = s["w"].double().view(co, 3, 3, ci).permute(0, 3, 1, 2).contiguous().requires_grad_(True)
    y = _conv64(x, W, s["b"].double())
    gx, gW = torch.autograd.grad(y, (x, W), image(s["g16"], co))
    rows = lambda v, c: v.detach().permute(0, 2, 3, 1).reshape(-1, c)
    return dict(y=rows(y, co), gx=rows(gx, ci), gw=gW.permute(0, 2, 3, 1).reshape(co, 9, ci), gb=s["g"].double().sum(0))


def exact(case, seed):
    return dict(sim=_exact_sim, batch=_exact_batch, train=_exact_train, warm=_exact_warm, conv=_exact_conv)[case["kind"]](
        case, seed)
