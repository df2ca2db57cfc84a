"""The forms a grid steps in, where the default of a small grid is the resident
step: the march by its own tiles with sliding walls against the oracle, and the
resident step against the march in every storage type and layout.

16-bit storage: both forms round every stored value once per step, and an FP32
difference of the last bit can turn a rounding by one unit of the stored value,
2^-11 (FP16) or 2^-8 (BF16) of it; 10 steps, at most 10 units: 5e-3 and 4e-2
normwise.  FP32 1e-5, FP64 1e-12, as in test_gpu_resident.  Without walls the two
forms are the same bits (with walls the compiler contracts some products apart)."""
import numpy as np
import pytest

from parity_helpers import normwise
from paper_1812_00118_gb300 import inputs as I
from test_gpu_moving_wall import CASES, run_case

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


TILES = {0: [(1, 16), (0, 5), (2, 7), (5, 4)], 1: [(8, 16), (1, 3), (3, 32), (9, 4)]}


@pytest.mark.parametrize("store", ["F64", "F32", "F16S"])
@pytest.mark.parametrize("case,tile", [(c, t) for c in (0, 1) for t in TILES[c]])
def test_sliding_walls_by_the_march(lbm, case, tile, store):
    lat_id, shape, bc, axis, walls = CASES[case]
    got, want, _ = run_case(lbm, lat_id, shape, bc, axis, walls, 40, tile=tile, store=getattr(lbm, store))
    tol = {"F64": 1e-10, "F32": 1e-5, "F16S": 2e-2}[store]
    for a, b in zip(got, want):
        assert normwise(a, b) < tol


FORMS = [((70, 45), (P, P)), ((31, 33), (W, P)), ((40, 37), (W, W)), ((13, 21, 17), (P, P, P)), ((19, 11, 25), (W, P, W))]


@pytest.mark.parametrize("band", [False, True])
@pytest.mark.parametrize("store", ["F64", "F32", "F16S", "BF16S"])
@pytest.mark.parametrize("shape,bc", FORMS)
def test_resident_against_the_march(lbm, shape, bc, store, band):
    L, dim = lbm, len(shape)
    nx, ny = shape[:2]
    nz = shape[2] if dim == 3 else 1
    phi, u, Pr = I.smooth_random((nz, ny, nx), 11, dim=dim, u_amp=0.01, P_amp=1e-4)
    prm = L.make_params(M=0.05, W=4.0, sigma=1e-3, rho_L=0.5, rho_H=1.0, nu_L=0.1, nu_H=0.1,
                        store=getattr(L, store), g=(1e-6, -2e-6, 0.0), g_scale=100.0 if store.endswith("S") else 0.0)
    sims = []
    for tile in (None, (1, 16)):
        s = L.Simulation(L.D2Q9 if dim == 2 else L.D3Q19, shape, prm, bc=bc, ghost_band=band)
        if tile:
            s.set_tile(*tile)
        for axis in range(dim):
            if bc[axis] == W:
                v = [0.01, -0.02, 0.005][:dim]
                v[axis] = 0.0
                s.set_wall_velocity(axis, 1, v)
        s.init_fields(*[np.ascontiguousarray(a.reshape(-1)) for a in (phi, u[:dim], Pr)])
        s.step(3)
        s.step(7)
        sims.append(s)
    tol = {"F64": 1e-12, "F32": 1e-5, "F16S": 5e-3, "BF16S": 4e-2}[store]
    errs = [normwise(a, b) for a, b in zip(sims[0].get_populations(), sims[1].get_populations())]
    print(shape, store, band, errs)
    assert max(errs) < tol
    if W not in bc:                        # without walls the forms round alike
        assert max(errs) == 0
    assert sims[0].diagnostics()["status"] == L.OK


def test_counts_start_over_freed_ones(lbm):
    """The counts of a context whose first state comes from lbm_set_populations,
    in memory that held the counts of smaller grids (the scratch of a context
    comes from the stream's memory pool)."""
    def state(shape):
        phi, u, Pr = I.smooth_random((1, shape[1], shape[0]), 5, dim=2, u_amp=0.01, P_amp=1e-4)
        return [np.ascontiguousarray(a.reshape(-1)) for a in (phi, u[:2], Pr)]
    prm = lbm.make_params(M=0.05, W=4.0, sigma=1e-3, rho_L=0.5, rho_H=1.0, nu_L=0.1, nu_H=0.1, store=lbm.F32)
    a = lbm.Simulation(lbm.D2Q9, (256, 192), prm)
    a.init_fields(*state((256, 192)))
    a.step(5)
    h, g = a.get_populations()
    a.step(20)
    want = a.get_populations()
    for small in ((64, 32), (32, 200), (150, 20)):
        for _ in range(4):
            s = lbm.Simulation(lbm.D2Q9, small, prm)
            s.init_fields(*state(small))
            s.step(37)
            s.close()
        b = lbm.Simulation(lbm.D2Q9, (256, 192), prm)
        b.set_populations(h, g)
        b.step(20)
        assert b.diagnostics()["status"] == lbm.OK
        for x, y in zip(b.get_populations(), want):
            assert np.array_equal(x, y)
        b.close()
