"""The resident step of small grids (one launch for many steps, boxes waiting
only for their neighbours) and the march fitted to one wave, against the same
steps through a tile the caller chose.

All forms compute the same arithmetic from the same device functions; compiled
apart they may contract a * b + c differently, so FP64 agrees to rounding
(1e-12 normwise after 38 steps of fields of O(1)) and FP32 to 1e-5, the stated
FP32 tolerance.  Many steps in one launch against one launch per step run the
same code: bit for bit."""
import numpy as np
import pytest

from paper_1812_00118_gb300 import inputs as I
from parity_helpers import normwise

pytestmark = pytest.mark.gpu
P, W = 0, 1


@pytest.fixture(scope="module")
def lbm():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1812_00118_gb300 import build, lbm as L
    build.build()
    L.load()
    return L


def make(L, shape, bc, store, tile=None, stream=None, fix=0):
    lat = L.D2Q9 if len(shape) == 2 else L.D3Q19
    nx, ny = shape[:2]
    nz = shape[2] if len(shape) == 3 else 1
    phi, u, Pr = I.smooth_random((nz, ny, nx), 11, dim=len(shape), u_amp=0.01, P_amp=1e-4)
    prm = L.make_params(M=0.05, W=4.0, sigma=1e-3, rho_L=0.5, rho_H=1.0, nu_L=0.1, nu_H=0.1, store=store,
                        g=(1e-6, -2e-6, 0.0), force_mode=1)
    sim = L.Simulation(lat, shape, prm, bc=bc, stream=stream)
    if tile is not None:
        sim.set_tile(*tile)
    if fix:
        sim.set_phi_correction(fix)
    sim.init_fields(np.ascontiguousarray(phi.reshape(-1)), np.ascontiguousarray(u[:len(shape)].reshape(-1)),
                    np.ascontiguousarray(Pr.reshape(-1)))
    return sim


SHAPES = [
    ((64, 64), (P, P)), ((33, 9), (P, P)), ((31, 33), (W, P)), ((150, 61), (P, W)), ((37, 50), (W, W)), ((1, 40), (P, P)),
    ((100, 1), (P, P)), ((3, 2), (W, P)), ((256, 256), (P, P)), ((512, 300), (P, W)),      # up to two boxes per CTA
    ((700, 700), (P, P)),                                                                   # the fitted march
    ((4, 64, 4), (P, W, P)), ((13, 21, 17), (P, P, P)), ((9, 9, 9), (W, W, W)), ((19, 11, 25), (W, P, W)),
    ((1, 1, 30), (P, P, P)), ((5, 1, 7), (P, P, W)), ((33, 30, 31), (P, P, P)), ((50, 47, 45), (P, P, W)),
]


@pytest.mark.parametrize("shape,bc", SHAPES)
@pytest.mark.parametrize("store", ["F64", "F32"])
def test_agrees_with_a_chosen_tile(lbm, shape, bc, store):
    a = make(lbm, shape, bc, getattr(lbm, store))
    b = make(lbm, shape, bc, getattr(lbm, store), (1, 16))
    tol = 1e-12 if store == "F64" else 1e-5
    for n in (1, 2, 35):
        a.step(n)
        b.step(n)
        for x, y in zip(a.get_populations(), b.get_populations()):
            assert normwise(x, y) < tol
    assert a.diagnostics()["status"] == lbm.OK


@pytest.mark.parametrize("shape,bc", [((256, 256), (P, P)), ((512, 300), (P, W)), ((40, 39, 37), (P, P, W)),
                                      ((17, 18, 19), (P, P, P))])
def test_one_launch_equals_single_steps(lbm, shape, bc):
    """64 steps in one launch (boxes waiting for each other) against 64 launches."""
    a, b = make(lbm, shape, bc, lbm.F32), make(lbm, shape, bc, lbm.F32)
    n0 = a.launch_count()
    a.step(64)
    assert a.launch_count() - n0 == 1
    for _ in range(64):
        b.step(1)
    for x, y in zip(a.get_populations(), b.get_populations()):
        assert np.array_equal(x, y)


def test_phi_correction_splits_the_launch(lbm):
    """A re-imposition every 5 steps falls between launches, at the steps it
    falls on with one launch per step."""
    a, b = make(lbm, (64, 48), (P, P), lbm.F16S, fix=5), make(lbm, (64, 48), (P, P), lbm.F16S, fix=5)
    a.step(13)
    a.step(4)
    for _ in range(17):
        b.step(1)
    for x, y in zip(a.get_populations(), b.get_populations()):
        assert np.array_equal(x, y)


def test_resume_without_initialisation(lbm):
    """A context whose first state comes from lbm_set_populations steps like the
    one the state came from (its box counts start at zero)."""
    import torch
    a = make(lbm, (256, 192), (P, P), lbm.F32)
    a.step(5)
    h, g = a.get_populations()
    junk = torch.full((1 << 22,), -1, dtype=torch.int32, device="cuda")   # what freed memory may hold
    del junk
    sims = []
    for _ in range(3):
        b = lbm.Simulation(lbm.D2Q9, (256, 192), a.params)
        b.set_populations(h, g)
        b.step(20)
        sims.append(b)
    a.step(20)
    want = a.get_populations()
    for b in sims:
        assert b.diagnostics()["status"] == lbm.OK
        for x, y in zip(b.get_populations(), want):
            assert np.array_equal(x, y)


def test_capture_and_replay(lbm):
    """A captured launch of 6 steps, replayed three times, equals 18 steps."""
    import torch
    s = torch.cuda.Stream()
    a, b = make(lbm, (96, 80), (P, P), lbm.F32, stream=s.cuda_stream), make(lbm, (96, 80), (P, P), lbm.F32)
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=s):
        a.step(6)
    for _ in range(3):
        g.replay()
    torch.cuda.synchronize()
    b.step(18)
    for x, y in zip(a.get_populations(), b.get_populations()):
        assert np.array_equal(x, y)


def test_two_streams_at_once(lbm):
    """Two grids stepped on two streams: both cooperative launches complete."""
    import torch
    ss = [torch.cuda.Stream() for _ in range(2)]
    sims = [make(lbm, (512, 300), (P, P), lbm.F32, stream=s.cuda_stream) for s in ss]
    ref = make(lbm, (512, 300), (P, P), lbm.F32)
    torch.cuda.synchronize()
    for _ in range(3):
        for s in sims:
            s.step(20)
    ref.step(60)
    want = ref.get_populations()
    for s in sims:
        for x, y in zip(s.get_populations(), want):
            assert np.array_equal(x, y)


def test_autotune_keeps_the_state(lbm):
    a, b = make(lbm, (64, 64), (P, P), lbm.F32), make(lbm, (64, 64), (P, P), lbm.F32)
    a.step(3)
    b.step(3)
    a.autotune(3)
    a.step(10)
    b.step(10)
    for x, y in zip(a.get_populations(), b.get_populations()):
        assert normwise(x, y) < 1e-5
