"""GPU parity of the small-grid direct simulations at the edges of their tiles: grids that
tiles do not fill, step counts that are not whole launches (odd ones copy back), the smallest
grids, and psi on grids that the synthesis tiles do not fill."""
import numpy as np
import pytest

from inputs import flows
import oracle
from tests._parity import rel_l2

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


def _flow(torch_mod, nf):
    spec = flows.cellular_two_scale(1.0 / 3, 1.0 / 3, 5)
    psi = torch_mod.tensor(oracle.grid_psi(spec, nf), dtype=torch_mod.float32, device="cuda:0")
    h = 2 * np.pi / nf
    return psi, psi.double().cpu().numpy(), 0.2 * min(h * h / 4, h / 2)


@pytest.mark.parametrize("nf,steps,prec", [(4, 3, "fp32"), (4, 3, "fp64"), (5, 9, "fp32"), (29, 2, "fp64"),
                                           (47, 5, "fp32"), (130, 4, "fp32"), (333, 3, "fp64"),
                                           (64, 1, "fp32"), (64, 1, "fp64"), (64, 0, "fp64")])
def test_dirichlet_edges(mlsd, torch_mod, nf, steps, prec):
    psi, psi_r, dt = _flow(torch_mod, nf)
    dtype = torch_mod.float64 if prec == "fp64" else torch_mod.float32
    U0 = flows.step_u0(nf) + 0.1 * flows.gaussian_u0(nf)
    u = torch_mod.tensor(U0, dtype=dtype, device="cuda:0")
    ut = torch_mod.empty_like(u)
    mlsd.dns_run_dirichlet(u, ut, psi, 1.0, dt, steps, 1.25, -0.5)
    ref = oracle.dns_run_dirichlet(psi_r, 1.0, dt, steps, U0, 1.25, -0.5)
    assert torch_mod.all(u[:, 0] == 1.25)
    assert rel_l2(u.cpu().numpy(), ref) < (1e-12 if prec == "fp64" else 1e-5)


@pytest.mark.parametrize("nf,steps", [(128, 1), (128, 7), (384, 9), (640, 4), (1024, 5)])
def test_periodic_edges(mlsd, torch_mod, monkeypatch, nf, steps):
    # the same cells as the per-tile kernel: equal to the bit
    psi, psi_r, dt = _flow(torch_mod, nf)
    u0 = torch_mod.tensor(flows.gaussian_u0(nf), dtype=torch_mod.float32, device="cuda:0")
    u, v, t = u0.clone(), u0.clone(), torch_mod.empty_like(u0)
    mlsd.dns_run(u, t, psi, 0.02, dt, steps)
    monkeypatch.setenv("MLSD_DNS_TY", "32")
    mlsd.dns_run(v, t, psi, 0.02, dt, steps)
    assert torch_mod.equal(u, v)


@pytest.mark.parametrize("nf", [1, 31, 100, 257])
def test_grid_psi_edges(mlsd, torch_mod, nf):
    spec = flows.continuous_spectrum(40, seed=3)
    g = torch_mod.zeros(nf, nf, dtype=torch_mod.float32, device="cuda:0")
    mlsd.grid_psi(spec, nf, g)
    ref = oracle.grid_psi(spec, nf)
    assert np.abs(g.cpu().numpy() - ref).max() < 1e-6 * np.abs(ref).max()
