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


@pytest.mark.parametrize("r,N", [(1, 5), (2, 3), (3, 4), (7, 9), (31, 2), (33, 3), (64, 3), (65, 2), (100, 1)])
@pytest.mark.parametrize("kind", ["normal", "cancelling", "wide", "denormal"])
def test_box_averages(mlsd, torch_mod, r, N, kind):
    # U against the exact sum of each box: one rounding to FP32, and the sum's own error, at most
    # half a unit of 2^-48 of the largest node per node (fixed point) or 2^-53 n of it (FP64)
    rng = np.random.default_rng(r)
    nf = r * N
    u = rng.standard_normal((nf, nf))
    if kind == "cancelling":
        u = 1e6 * (u - u.mean()) + 1.0
    if kind == "wide":
        u *= 10.0 ** rng.uniform(-30, 5, u.shape)
    if kind == "denormal":
        u *= 1e-40
    u = u.astype(np.float32)
    U = torch_mod.full((N, N), 7.0, dtype=torch_mod.float32, device="cuda:0")
    m = mlsd.coarse_grain(torch_mod.tensor(u, device="cuda:0"), N, U)
    ul = np.roll(u.astype(np.longdouble), (r // 2, r // 2), (0, 1)).reshape(N, r, N, r)
    box, top = ul.sum((1, 3)), np.abs(ul).max((1, 3))
    ref = box / (r * r)
    tol = np.abs(ref) * 2.0**-24 * 1.01 + top * 2.0**-38 * 2.0**-10 + 2.0**-150
    assert np.all(np.abs(U.cpu().numpy() - ref) <= tol)
    h = 2 * np.pi / nf
    assert abs(m - box.sum() * h * h) <= h * h * nf * nf * float(top.max()) * 2.0**-46


@pytest.mark.parametrize("r", [4, 65])
def test_box_averages_not_finite(mlsd, torch_mod, r):
    # boxes reach half a side back: node (0, 0) and node (r, 2 r) are inside boxes (0, 0) and (1, 2)
    u = torch_mod.ones(3 * r, 3 * r, dtype=torch_mod.float32, device="cuda:0")
    u[0, 0], u[r, 2 * r], u[r, 0], u[r, 1] = float("nan"), float("-inf"), float("inf"), float("-inf")
    U = torch_mod.empty(3, 3, dtype=torch_mod.float32, device="cuda:0")
    mlsd.coarse_grain(u, 3, U, want_mass=False)
    V = U.cpu().numpy()
    assert np.isnan(V[0, 0]) and V[1, 2] == -np.inf and np.isnan(V[1, 0])
    assert np.all(V[[0, 0, 1, 2, 2, 2], [1, 2, 1, 0, 1, 2]] == 1.0)


def test_dirichlet_without_coefficients(mlsd, torch_mod):
    # above 8192^2 the FP64 steps form their coefficients themselves: the same operations as on
    # smaller grids.  psi and u do not depend on x2 (v2 = 0 exactly, v1 = 0), so each row is the
    # heat equation of a 1-D row: the sum of the same five terms, some 10 roundings of O(1) values
    nf, steps, dt, kappa = 8193, 2, 1e-8, 0.7
    h = 2 * np.pi / nf
    x = np.arange(nf) * h
    row = np.cos(3 * x) + 1.5
    u = torch_mod.tensor(row, dtype=torch_mod.float64, device="cuda:0").repeat(nf, 1).contiguous()
    ut = torch_mod.empty_like(u)
    psi = torch_mod.full((nf, nf), 0.25, dtype=torch_mod.float32, device="cuda:0")
    mlsd.dns_run_dirichlet(u, ut, psi, kappa, dt, steps, 2.5, 2.5)
    ref = row.copy()
    ref[0] = 2.5

    def f(v):
        e = np.append(v, 2.5)
        g = np.zeros_like(v)
        g[1:] = kappa * (e[2:] - 2 * e[1:-1] + e[:-2]) / (h * h)
        return g
    for _ in range(steps):
        k1 = f(ref)
        ref = ref + dt / 2 * (k1 + f(ref + dt * k1))
    got = u.cpu().numpy()
    assert np.max(np.abs(got[[0, 1, 4000, nf - 1]] - ref)) <= 40 * 2.0**-52 * 2.5
    assert np.array_equal(got[4000], got[17]) or np.max(np.abs(got[4000] - got[17])) <= 40 * 2.0**-52 * 2.5


@pytest.mark.parametrize("nf,prec", [(512, "fp32"), (512, "fp64"), (2048, "fp32")])
def test_captured_runs(mlsd, torch_mod, nf, prec):
    # a captured run, replayed on new values of the same buffers, gives the direct call's bits
    psi, _, dt = _flow(torch_mod, nf)
    dtype = torch_mod.float64 if prec == "fp64" else torch_mod.float32
    u0 = torch_mod.tensor(flows.gaussian_u0(nf), dtype=dtype, device="cuda:0")
    u, ut = u0.clone(), torch_mod.empty_like(u0)

    def step():
        if prec == "fp64":
            mlsd.dns_run_dirichlet(u, ut, psi, 1.0, dt, 5, 1.0, 0.0)
        else:
            mlsd.dns_run(u, ut, psi, 1.0, dt, 5)
    step()
    ref = u.clone()
    u.copy_(u0)
    g = torch_mod.cuda.CUDAGraph()
    with torch_mod.cuda.graph(g):
        step()
    assert torch_mod.equal(u, u0)
    g.replay()
    torch_mod.cuda.synchronize()
    assert torch_mod.equal(u, ref)
