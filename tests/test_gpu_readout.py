"""lbm_macro writes device outputs in place: the same values as the host path,
any subset of outputs, and outputs that overlap one another; phi is the sum of
the populations to FP64 rounding for every storage type."""
import math

import numpy as np
import pytest

from paper_1812_00118_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lbm():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1812_00118_gb300 import build, lbm as L
    build.build()
    L.load()
    return L


def state(L, shape, bc, store):
    lat = L.D2Q9 if len(shape) == 2 else L.D3Q19
    nx, ny = shape[:2]
    nz = shape[2] if len(shape) == 3 else 1
    phi, u, P = I.smooth_random((nz, ny, nx), 21, dim=len(shape))
    prm = L.make_params(M=0.05, W=4.0, sigma=1e-3, rho_L=0.1, rho_H=1.0, nu_L=0.1, nu_H=0.1, store=store,
                        g_scale=100.0 if store == L.F16S else 0.0, g=(1e-6, 0.0, 0.0))
    sim = L.Simulation(lat, shape, prm, bc=bc)
    sim.init_fields(np.ascontiguousarray(phi.reshape(-1)), np.ascontiguousarray(u[:len(shape)].reshape(-1)),
                    np.ascontiguousarray(P.reshape(-1)))
    sim.step(3)
    return sim


@pytest.mark.parametrize("shape,bc", [((33, 17), (0, 1)), ((9, 13, 7), (0, 0, 1)), ((70, 5, 31), (1, 0, 0))])
@pytest.mark.parametrize("store", ["F64", "F32", "F16S"])
def test_device_outputs(lbm, shape, bc, store):
    import torch
    sim = state(lbm, shape, bc, getattr(lbm, store))
    host = sim.macro()
    z = lambda k: torch.full((k,), 7.0, dtype=torch.float64, device="cuda")
    N, dim = sim.N, sim.dim
    for want in [(1, 1, 1), (1, 0, 0), (0, 1, 0), (0, 0, 1), (1, 1, 0), (0, 1, 1)]:
        out = [z(k) if w else None for w, k in zip(want, (N, N, dim * N))]
        sim.macro(*out)
        for o, h in zip(out, host):
            if o is not None:
                assert np.array_equal(o.cpu().numpy(), h)
    # outputs over one another: the last one written stays, as with separate copies
    both = z(N)
    sim.macro(both, both)
    assert np.array_equal(both.cpu().numpy(), host[1])
    wide = z((dim + 1) * N)
    sim.macro(wide[:N], None, wide[N // 2:N // 2 + dim * N])
    w = wide.cpu().numpy()
    assert np.array_equal(w[:N // 2], host[0][:N // 2])
    assert np.array_equal(w[N // 2:N // 2 + dim * N], host[2])


@pytest.mark.parametrize("store", ["F64", "F32", "F16S"])
def test_phi_is_the_sum_of_h(lbm, store):
    sim = state(lbm, (24, 20, 12), (0, 0, 1), getattr(lbm, store))
    phi = sim.macro()[0]
    h = sim.get_populations()[0].reshape(sim.Q, sim.N)
    exact = np.array([math.fsum(h[:, n]) for n in range(sim.N)])
    # one FP64 rounding of the sum, or the 18 of a chain with FP64 storage
    assert np.abs(phi - exact).max() <= (20 if store == "F64" else 1) * 2.0 ** -53


def test_not_finite_stays_not_finite(lbm):
    sim = state(lbm, (16, 16, 16), (0, 0, 0), lbm.F32)
    h, g = sim.get_populations()
    for bad in (np.inf, -np.inf, np.nan):
        k = h.copy()
        k[5 * sim.N + 100] = bad
        sim.set_populations(k, g)
        phi = sim.macro()[0]
        assert np.isfinite(np.delete(phi, 100)).all()
        assert phi[100] == bad or (np.isnan(bad) and np.isnan(phi[100]))
        assert sim.diagnostics(raise_on_divergence=False)["nonfinite"] >= 1


def test_device_outputs_on_any_address(lbm):
    """Device outputs that do not start on 8-byte boundaries are copied to, as they
    were when every output was a copy."""
    import ctypes

    import torch
    sim = state(lbm, (33, 17), (0, 1), lbm.F32)
    host = sim.macro()
    lib, N = lbm.load(), sim.N
    for k in range(3):                    # one odd output at a time, then all three
        offs = [[4, 0, 0], [0, 0, 1], [4, 2, 12]][k]
        bufs = [torch.zeros(8 * n + 16, dtype=torch.uint8, device="cuda") for n in (N, N, 2 * N)]
        ptrs = [ctypes.c_void_p(b.data_ptr() + o) for b, o in zip(bufs, offs)]
        assert lib.lbm_macro(sim.ctx, *ptrs, 1) == lbm.OK
        for b, o, h in zip(bufs, offs, host):
            got = np.frombuffer(b.cpu().numpy()[o:o + 8 * h.size].tobytes(), dtype=np.float64)
            assert np.array_equal(got, h)
