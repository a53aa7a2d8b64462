"""Calls at the edges of what the entry points accept."""
import math
import subprocess
import sys

import numpy as np
import pytest

from inputs import flows
from tests.conftest import ROOT

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


def test_macro_past_32_bit_coefficients(mlsd, torch_mod):
    # 4 N^2 > 2^31 - 1: the face coefficients of the last cells lie past a 32-bit index.  K and U
    # depend on x1 only, so every row is the same 1-D problem: Heun in FP64 on the host against a few
    # FP32 roundings of O(1) values
    N, steps = 23171, 2
    if torch_mod.cuda.mem_get_info()[0] < 40 << 30:
        pytest.skip("needs 40 GB")
    H = 2 * np.pi / N
    x = np.arange(N) * H
    k = 1.0 + 0.5 * np.cos(5 * x)
    row = 1.5 + np.cos(3 * x)
    dt = 0.1 * H * H
    K = torch_mod.zeros(N, N, 3, dtype=torch_mod.float64, device="cuda:0")
    K[:, :, 0] = torch_mod.tensor(k, device="cuda:0")
    K[:, :, 2] = 0.75
    U = torch_mod.tensor(row, dtype=torch_mod.float32, device="cuda:0").repeat(N, 1)
    mlsd.macro_step(U, K, dt, steps, want_mass=False)
    kf = 0.5 * (k + np.roll(k, -1)) * dt / (H * H)

    def f(u):
        flux = kf * (np.roll(u, -1) - u)
        return flux - np.roll(flux, 1)
    ref = row
    for _ in range(steps):
        s = ref + f(ref)
        ref = 0.5 * (ref + s + f(s))
    for j in (0, 1, N // 2, N - 2, N - 1):
        assert np.abs(U[j].double().cpu().numpy() - ref).max() < 20 * 2.0**-24 * 2.5
    assert torch_mod.equal(U[0], U[N - 1]) and bool((U == U[0]).all())


@pytest.mark.parametrize("n", [32, 64])
@pytest.mark.parametrize("xo,fo", [(1, 0), (0, 1), (3, 3), (2, 2)])
def test_feature_rows_at_any_offset(mlsd, torch_mod, n, xo, fo):
    # X and F32 need the alignment of their elements only
    lv = mlsd.Levels(flows.cellular_two_scale(0.8, 0.5, 4), 0.03, 3, [1, 4, 8], [n, n],
                     n_burn_fixed=0, n_avg_fixed=4)
    B = torch_mod.tensor([[0.05, 0.01, 0.04]] * 9, dtype=torch_mod.float64, device="cuda:0")

    def rows(xo, fo):
        X = torch_mod.full((9 * mlsd.SUR_IN + 8,), -7.0, dtype=torch_mod.bfloat16, device="cuda:0")
        F = torch_mod.full((9 * mlsd.SUR_FEATURES + 8,), -7.0, device="cuda:0")
        x, f = X[xo:xo + 9 * mlsd.SUR_IN], F[fo:fo + 9 * mlsd.SUR_FEATURES]
        lv.features(2, B, x, f)
        outside = torch_mod.cat([X[:xo].float(), X[xo + len(x):].float(), F[:fo], F[fo + len(f):]])
        assert bool((outside == -7.0).all())
        return x.clone(), f.clone()
    x0, f0 = rows(0, 0)
    x1, f1 = rows(xo, fo)
    assert torch_mod.equal(x0, x1) and torch_mod.equal(f0, f1)
    # the data set's rows come from the same kernel
    X = torch_mod.empty(9 * mlsd.SUR_IN + 8, dtype=torch_mod.bfloat16, device="cuda:0")[xo:xo + 9 * mlsd.SUR_IN]
    Y = torch_mod.empty(9, 3, device="cuda:0")
    lv.surrogate_dataset(2, B, X, Y)
    assert torch_mod.equal(X, x0)


@pytest.mark.parametrize("r", [4, 16, 32, 64, 100])
@pytest.mark.parametrize("kind", ["one large", "cancelling", "spread", "denormal"])
def test_box_sums_of_unequal_nodes(mlsd, torch_mod, r, kind):
    # the box's sum in FP64: no worse than adding its nodes one by one in a tree of the kernel's
    # depth (16 nodes a lane, 5 levels of a warp, 8 warps, a chunk after the other), each addition
    # off by half a unit of the sum of the magnitudes at most
    rng = np.random.default_rng(r)
    u = np.full((r, r), 3e-15) * rng.uniform(0.5, 1.5, (r, r))
    if kind == "one large":
        u[r // 2, 1] = 1.0
    if kind == "cancelling":
        u[r // 2, 1], u[0, r - 1] = 1.0, -1.0
    if kind == "spread":
        u = rng.standard_normal((r, r)) * 10.0 ** rng.uniform(-30, 5, (r, r))
    if kind == "denormal":
        u = rng.standard_normal((r, r)) * 2.0 ** rng.uniform(-148, -60, (r, r))
    u = u.astype(np.float32)
    U = torch_mod.empty(1, 1, dtype=torch_mod.float32, device="cuda:0")
    m = mlsd.coarse_grain(torch_mod.tensor(u, device="cuda:0"), 1, U)
    exact, mag = math.fsum(u.ravel().astype(float)), math.fsum(np.abs(u.ravel().astype(float)))
    depth = 16 + 5 + 8 + (r * r + 4095) // 4096
    h2 = (2 * np.pi / r) ** 2
    assert abs(m / h2 - exact) <= (depth + 4) * 2.0**-53 * mag
    mean = exact / (r * r)
    assert abs(float(U) - mean) <= abs(mean) * 2.0**-24 * 1.01 + depth * 2.0**-53 * mag / (r * r) + 2.0**-150
    # whole boxes of the same kind beside narrow ones
    v = np.tile(u, (3, 3))
    v[:r, :r] = 0.5
    V = torch_mod.empty(3, 3, dtype=torch_mod.float32, device="cuda:0")
    v = np.roll(v, (-(r // 2), -(r // 2)), (0, 1))
    mlsd.coarse_grain(torch_mod.tensor(v, device="cuda:0"), 3, V, want_mass=False)
    V = V.cpu().numpy()
    assert V[0, 0] == 0.5 and np.all(np.abs(V.ravel()[1:] - mean) <=
                                     abs(mean) * 2.0**-24 * 1.01 + depth * 2.0**-53 * mag / (r * r) + 2.0**-150)


def _dns(torch_mod, nf):
    spec = flows.cellular_two_scale(1.0 / 3, 1.0 / 3, 5)
    import paper_1510_00451_gb300 as m
    psi = torch_mod.empty(nf, nf, dtype=torch_mod.float32, device="cuda:0")
    m.grid_psi(spec, nf, psi)
    h = 2 * np.pi / nf
    u0 = torch_mod.tensor(flows.gaussian_u0(nf), dtype=torch_mod.float32, device="cuda:0")
    return psi, u0, 0.2 * min(h * h / 4, h / 2)


@pytest.mark.parametrize("pin,name", [("t32", "k_dns_tma<32,1>"), ("t32x2", "k_dns_tma<32,2>"),
                                      ("t64", "k_dns_tma<64,1>"), ("t32p", "k_dns_tma<32,1,pairs>"),
                                      ("32", "k_dns_step<32>")])
@pytest.mark.parametrize("steps", [1, 4, 5])
def test_captured_dns_replays(mlsd, torch_mod, monkeypatch, pin, name, steps):
    # every replay of a captured run gives the direct run's bits, whatever ran before it
    monkeypatch.setenv("MLSD_DNS_TY", pin)
    nf = 512
    psi, u0, dt = _dns(torch_mod, nf)
    u, ut = u0.clone(), torch_mod.empty_like(u0)
    v, vt = u0.clone(), torch_mod.empty_like(u0)
    mlsd.dns_run(u, ut, psi, 0.02, dt, steps)
    assert mlsd.dns_kernel() == name
    ref = u.clone()
    assert not torch_mod.equal(ref, u0)
    g = torch_mod.cuda.CUDAGraph()
    with torch_mod.cuda.graph(g):
        mlsd.dns_run(u, ut, psi, 0.02, dt, steps)
    mlsd.dns_run(v, vt, psi, 0.02, dt, 3)
    for k in range(4):
        u.copy_(u0)
        ut.fill_(float("nan"))
        g.replay()
        assert torch_mod.equal(u, ref), k
        if k == 2:
            v.copy_(u0)
            vt.fill_(float("nan"))
            mlsd.dns_run(v, vt, psi, 0.02, dt, steps)
            assert torch_mod.equal(v, ref)
    assert mlsd.dns_status() == 0


def test_pinned_dns_kernel_is_not_kept(mlsd, torch_mod, monkeypatch):
    # a pin chooses the kernel of the runs it is set for; the timed choice stays
    monkeypatch.delenv("MLSD_DNS_TY", raising=False)
    psi, u, dt = _dns(torch_mod, 1152)
    ut = torch_mod.empty_like(u)
    mlsd.dns_run(u, ut, psi, 0.02, dt, 1)
    chosen = mlsd.dns_kernel()
    for pin, name in (("64", "k_dns_step<64>"), ("32", "k_dns_step<32>"), ("t32", "k_dns_tma<32,1>")):
        monkeypatch.setenv("MLSD_DNS_TY", pin)
        mlsd.dns_run(u, ut, psi, 0.02, dt, 1)
        assert mlsd.dns_kernel() == name
        monkeypatch.delenv("MLSD_DNS_TY")
        mlsd.dns_run(u, ut, psi, 0.02, dt, 1)
        assert mlsd.dns_kernel() == chosen


def test_first_large_dns_run_is_captured(torch_mod):
    # a program that ran a small grid may capture its first large one: no kernel is timed under
    # capture (a process of its own: the choice is made once per process)
    code = """
import numpy as np, torch
import paper_1510_00451_gb300 as m
from inputs import flows
def case(nf):
    psi = torch.empty(nf, nf, device='cuda:0')
    m.grid_psi(flows.cellular_two_scale(1.0 / 3, 1.0 / 3, 5), nf, psi)
    u0 = torch.tensor(flows.gaussian_u0(nf), dtype=torch.float32, device='cuda:0')
    h = 2 * np.pi / nf
    return psi, u0, torch.empty_like(u0), 0.2 * min(h * h / 4, h / 2)
psi, u, ut, dt = case(256)
m.dns_run(u, ut, psi, 0.02, dt, 3)
psi, u0, ut, dt = case(1152)
u = u0.clone()
g = torch.cuda.CUDAGraph()
torch.cuda.synchronize()
with torch.cuda.graph(g):
    m.dns_run(u, ut, psi, 0.02, dt, 3)
assert torch.equal(u, u0)
for k in range(2):
    u.copy_(u0)
    g.replay()
    v = u0.clone()
    m.dns_run(v, ut, psi, 0.02, dt, 3)
    torch.cuda.synchronize()
    assert float((u - v).abs().max()) <= 1e-6 and float((u - u0).abs().max()) > 1e-6
print('captured')
"""
    out = subprocess.run([sys.executable, "-c", code], cwd=ROOT, capture_output=True, text=True, timeout=300)
    assert out.returncode == 0 and "captured" in out.stdout, out.stderr[-2000:]


def test_macro_workspace_without_mass(mlsd, torch_mod):
    # without the mass record the workspace does not grow with the number of steps: it would be
    # 86 MB here.  The memory is the pool's until the next synchronisation, in pieces of 32 MB
    N, steps = 33, 1200000
    U = torch_mod.ones(N, N, dtype=torch_mod.float32, device="cuda:0")
    K = torch_mod.ones(N * N, 3, dtype=torch_mod.float64, device="cuda:0")
    mlsd.macro_step(U, K, 1e-4, 5, want_mass=False)
    mlsd.Surrogate(1, 32, 8).close()                    # gives the pool's idle memory back
    before = torch_mod.cuda.mem_get_info()[0]
    mlsd.macro_step(U, K, 1e-4, steps, want_mass=False)
    after = torch_mod.cuda.mem_get_info()[0]
    torch_mod.cuda.synchronize()
    assert before - after < 64 << 20
    assert bool((U == 1.0).all())


@pytest.mark.parametrize("k1,k2", [(-2**31, 3), (3, -2**31), (2**31 - 1, -5), (-2**31 + 1, 2), (0, -2**31)])
def test_grid_psi_wave_numbers_of_any_int(mlsd, torch_mod, k1, k2):
    # a point's phase is (k1 x + k2 y) mod nf: exact in integers, whatever the wave numbers
    class Spec:
        def as_arrays(self):
            return (np.array([k1], np.int32), np.array([k2], np.int32), np.array([0.75]), np.array([-0.5]))
    nf = 7
    g = torch_mod.zeros(nf, nf, dtype=torch_mod.float32, device="cuda:0")
    mlsd.grid_psi(Spec(), nf, g)
    y, x = np.mgrid[:nf, :nf]
    ph = 2 * np.pi * (((k1 % nf) * x + (k2 % nf) * y) % nf) / nf
    assert np.abs(g.cpu().numpy() - (0.75 * np.cos(ph) + 0.5 * np.sin(ph))).max() < 4 * 2.0**-24
