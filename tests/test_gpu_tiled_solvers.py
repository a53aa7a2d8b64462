"""GPU parity of the macro solver at the edges of its kernels: the largest grids of the
resident kernel and the smallest of the tiled one, tiles that the grid does not fill, step
counts that are not whole launches, and the mass record of each."""
import numpy as np
import pytest

from inputs import flows
import oracle
from tests._parity import rel_l2, random_spd

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch_mod():
    import torch
    assert torch.cuda.is_available()
    return torch


@pytest.fixture(scope="module")
def mlsd():
    import paper_1510_00451_gb300 as m
    return m


@pytest.mark.parametrize("N,steps,prec", [(2, 3, "fp32"), (3, 5, "fp64"), (16, 7, "fp64"), (17, 6, "fp64"),
                                          (32, 9, "fp32"), (33, 1, "fp32"), (33, 4, "fp32"), (47, 13, "fp32"),
                                          (129, 6, "fp64"), (130, 10, "fp32")])
def test_macro_edges(mlsd, torch_mod, N, steps, prec):
    # the bounds of the solver's other parity tests: FP32 rounding of a few steps, FP64 rounding
    tol, mtol = (1e-12, 1e-13) if prec == "fp64" else (1e-5, 1e-6)
    dtype = torch_mod.float64 if prec == "fp64" else torch_mod.float32
    K = random_spd(N * N, np.random.default_rng(N), 0.1, 1.0)
    U0 = 0.5 + flows.gaussian_u0(N)
    dt = oracle.macro_dt(K, N, 0.2)
    Kg = torch_mod.tensor(K, dtype=torch_mod.float64, device="cuda:0")
    U = torch_mod.tensor(U0, dtype=dtype, device="cuda:0")
    V = U.clone()
    mass = mlsd.macro_step(U, Kg, dt, steps)
    Ur, mr = oracle.macro_run(U0, K, dt, steps)
    assert rel_l2(U.cpu().numpy(), Ur) < tol
    assert len(mass) == steps + 1 and np.max(np.abs(mass / mr - 1)) < max(mtol, 1e-7 if prec == "fp32" else 0)
    mlsd.macro_step(V, Kg, dt, steps, want_mass=False)
    assert torch_mod.equal(U, V)
    W = torch_mod.tensor(U0, dtype=dtype, device="cuda:0")
    mlsd.macro_step_dirichlet(W, Kg, dt, steps, 1.25, -0.5)
    Wr = oracle.macro_run_dirichlet(U0, K, dt, steps, 1.25, -0.5)
    assert torch_mod.all(W[:, 0] == 1.25)
    assert rel_l2(W.cpu().numpy(), Wr) < tol


@pytest.mark.parametrize("n,tile", [(32, "4x4"), (32, "2x4"), (32, "4x4p"), (64, "4x8m3"), (64, "4x4p")])
def test_no_cross_term_is_the_same(mlsd, torch_mod, monkeypatch, n, tile):
    # B12 = 0 leaves the cross term out; a B12 so small that its products vanish against
    # every sum keeps it and has to give the same bits
    monkeypatch.setenv("MLSD_TILE", tile)
    lv = mlsd.Levels(flows.cellular_two_scale(0.8, 0.5, 4), 0.03, 3, [1, 4, 8], [n, n],
                     n_burn_fixed=40, n_avg_fixed=35)
    B = random_spd(9, np.random.default_rng(n), 0.03, 0.1)
    out = []
    for b12 in (0.0, 1e-30):
        B[:, 1] = b12
        Kb = torch_mod.tensor(B, dtype=torch_mod.float64, device="cuda:0")
        K, w = torch_mod.zeros_like(Kb), torch_mod.zeros(9, 2, n, n, device="cuda:0")
        lv.solve_level(2, Kb, K, w)
        assert lv.status() == 0
        out.append((K, w))
    assert torch_mod.equal(out[0][1], out[1][1])
    assert torch_mod.equal(out[0][0][:, ::2], out[1][0][:, ::2])
