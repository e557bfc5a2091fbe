"""Kernels that no other test launches, against the FP64 oracle: the complex form of the cavity-structure fibers and the
plain fibers (given tile widths; automatic ones take smaller mappings at these sizes), the cluster kernel of
two-node density matrices in FP32, at its largest size and per interval, the strided gradient and the reverse
gradient in FP64 at d = 6561.  test_routes_host.py shows that these problems launch these kernels.  Tolerances are those of
test_gpu_parity.py, test_gpu_density.py and test_gpu_gradient.py for the same quantities."""
import cmath
import functools

import numpy as np
import pytest

import synth_inputs as si
from oracle import density as od
from oracle import gradient as og
from oracle import mcwf
from oracle import model as om
from paper_1801_04382_gb300 import DensityProblem, Problem, cascaded_chain
from test_gpu_parity import compare, setup

pytestmark = pytest.mark.gpu

G = cmath.exp(0.2j * cmath.pi)


def models(kind, N, nc):
    """The library's network and the oracle's model: a coupling with a phase, or a real coupling (e, n) <-> (g, n) that the
    cavity structure does not have."""
    if kind == "complex":
        return cascaded_chain(N, nc, g=G), om.build_model(N, nc, g=G)
    net, m = cascaded_chain(N, nc), om.build_model(N, nc)
    nl, NP = net.n_loc, nc + 1
    x = np.zeros((nl, nl), dtype=np.complex128)
    for n in range(NP):
        x[n, NP + n] = x[NP + n, n] = 0.4
    net.h0_local = net.h0_local + x
    for i in range(N):
        m.H0 = m.H0 + om.embed(x, i, N)
    return net, m


@functools.lru_cache(maxsize=None)
def fiber_case(kind, nc):
    nt, M = (12, 5) if nc == 1 else (6, 3)
    c = setup(2, nc, 0.05 * nt, nt, M, 30.0, 7, 1, random_init=True)
    net, m = models(kind, 2, nc)
    return c, net, m, mcwf.optimize(m, c["eps0"], c["T"], c["U"], c["S"], c["lam"], 1, psi0=c["psi0"], keep=True)


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("kind,nc,tile", [("complex", 1, 1), ("complex", 1, 4), ("complex", 2, 1), ("complex", 2, 2),
                                          ("plain", 1, 2), ("plain", 2, 1)])
def test_general_fibers(kind, nc, tile, precision, monkeypatch):
    c, net, m, res = fiber_case(kind, nc)
    monkeypatch.setattr(om, "build_model", lambda *a, **k: m)      # compare() replays FP32 records in the oracle's model
    out = {"F": [], "recs": [], "psiT": [], "eps": [], "deps": [], "tau": []}
    with Problem(net, c["T"], c["nt"], c["M"], c["eps0"], c["S"], c["lam"], c["U"], psi0_batch=c["psi0"], precision=precision,
                 tile_traj=tile) as p:
        assert p.info.items_per_thread == 0 and p.info.tile_traj == tile
        for it in range(2):
            if it:
                p.backward()
            out["F"].append(p.forward(it > 0))
            out["tau"].append(p.fidelity()[1])
            out["recs"].append(p.records())
            out["psiT"].append(p.states())
            if it:
                out["eps"].append(p.pulses())
                out["deps"].append(p.deps())
    assert sum(len(r) for r in out["recs"][0] + out["recs"][1]) >= 1
    if precision == "fp64":
        compare(c, out, res, 1e-10, 1e-10, 1e-10, 1e-9)
    else:
        compare(c, out, res, 3e-5, 1e-5, 1e-4, 1e-4, margin_min=1e-5)


def density_step(m, eps, X, dt, adjoint=False):
    """exp(dt L) of a density matrix, or exp(dt L^dag) of a co-state, as Taylor series over steps of norm one:
    the oracle's dense exponential of the Liouville-space map takes minutes at d^2 = 6561."""
    H = m.Heff(eps)
    n = int(np.ceil(2.0 * np.linalg.norm(H, 2) * dt))
    out = X
    for _ in range(n):
        t, k = out, 0
        while np.abs(t).max() > 1e-18:
            k += 1
            if adjoint:
                t = 1j * (H.conj().T @ t - t @ H) + sum(l.conj().T @ t @ l for l in m.L)
            else:
                t = -1j * (H @ t - t @ H.conj().T) + sum(l @ t @ l.conj().T for l in m.L)
            t = t * (dt / n / k)
            out = out + t
    return out


def test_density_step_is_the_oracles():
    m = om.build_model(1, 2)
    eps, rho = np.full((1, 2), 3.0), np.outer(m.psi0, m.psi0.conj())
    P = od.backward_P(m, eps, 0.4, np.outer(m.psi_tgt, m.psi_tgt.conj()))
    assert np.abs(density_step(m, eps[:, 0], P[2], 0.2, adjoint=True) - P[1]).max() <= 1e-12
    _, _, rho_T = od.forward_update(m, eps, 0.4, rho, P, np.zeros((1, 2)), np.ones(1))
    assert np.abs(density_step(m, eps[:, 1], density_step(m, eps[:, 0], rho, 0.2), 0.2) - rho_T).max() <= 1e-12


@pytest.mark.parametrize("nc,nt,precision", [(1, 6, "fp32"), (2, 3, "fp64"), (2, 3, "fp32")])
def test_density_cluster(nc, nt, precision):
    """One Krotov iteration of two nodes: as whole sweeps, with one launch per interval and with checkpointed
    co-states, which agree bit for bit."""
    T = 0.1 * nt if nc == 1 else 0.05 * nt
    m = om.build_model(2, nc)
    eps0, S, lam = si.guess_pulses(2, nt, T, 20.0), si.shape_functions(2, nt, T), np.full(2, 2.0)
    dt, rho = T / nt, np.outer(m.psi0, m.psi0.conj())
    P = [None] * nt + [np.outer(m.psi_tgt, m.psi_tgt.conj())]
    rho_0 = rho
    for j in range(nt):
        rho_0 = density_step(m, eps0[:, j], rho_0, dt)
    F0 = 1.0 - od.functional(m, rho_0)
    for j in range(nt - 1, -1, -1):
        P[j] = density_step(m, eps0[:, j], P[j + 1], dt, adjoint=True)
    deps, rho_T = np.zeros_like(eps0), rho
    for j in range(nt):
        for i, h in enumerate(m.Hc):
            deps[i, j] = S[i, j] / lam[i] * np.imag(np.trace(P[j].conj().T @ (h @ rho_T - rho_T @ h)))
        rho_T = density_step(m, eps0[:, j] + deps[:, j], rho_T, dt)
    got = []
    for more in ({}, {"per_interval_launches": True}, {"ckpt_interval": 2}):
        with DensityProblem(cascaded_chain(2, nc), T, nt, eps0, S, lam, precision=precision, **more) as p:
            assert p.info.whole_sweep == (not more)
            g0 = p.forward(False)
            p.backward()
            P0 = p.P(0)
            g1 = p.forward(True)
            got.append((g0, g1, P0, p.deps(), p.rho()))
    tol, tol_F = (1e-10, 1e-10) if precision == "fp64" else (1e-4, 1e-5)
    g0, g1, P0, g_deps, g_rho = got[0]
    assert abs(g0 - F0) <= tol_F and abs(g1 - (1.0 - od.functional(m, rho_T))) <= tol_F
    assert np.abs(P0 - P[0]).max() <= tol * np.abs(P[0]).max()
    assert np.abs(g_deps - deps).max() <= tol * np.abs(deps).max()
    assert np.abs(g_rho - rho_T).max() <= tol * np.abs(rho_T).max()
    for other in got[1:]:
        assert all(np.array_equal(a, b) for a, b in zip(got[0], other))


@pytest.mark.parametrize("precision,tol", [("fp64", 1e-10), ("fp32", 2e-4)])
def test_strided_gradient(precision, tol):
    N, nc, M, nt, T = 2, 1, 4, 24, 1.2
    eps, S = si.guess_pulses(N, nt, T, 30.0), si.shape_functions(N, nt, T)
    U, psi0 = si.uniforms(5, 2, M, 1 + 2 * N * (1 + nc)), si.random_states(55, M, 36)
    net, m = models("complex", N, nc)
    with Problem(net, T, nt, M, eps, S, np.full(N, 10.0), U, psi0_batch=psi0, precision=precision) as p:
        p.forward(keep_for_gradient=True)
        recs = p.records()
        grad = p.gradient().cpu().numpy()
    assert sum(len(r) for r in recs) >= 1
    ref, _ = og.gradient(m, eps, T, psi0, [[mcwf.Jump(*r) for r in rk] for rk in recs])
    assert np.abs(grad - ref).max() <= tol * np.abs(ref).max()


def test_gradient_fp64_d6561_matches_central_differences():
    """No jump; h = 0.05 changes the phase of an interval by 5e-4, so the differences are off by its square, 3e-7
    relative, and by 1e-15 / h."""
    N, nc, M, nt, dt, h = 4, 2, 2, 3, 0.01, 0.05
    eps, S = si.guess_pulses(N, nt, nt * dt, 2.0), si.shape_functions(N, nt, nt * dt)
    net = cascaded_chain(N, nc)
    psi0 = si.random_states(3, M, net.d) + 0.7 * net.psi_tgt
    psi0 /= np.linalg.norm(psi0, axis=1, keepdims=True)
    U = np.full((1, M, 1 + 2 * N * (nc + 1)), 1e-9)
    with Problem(net, nt * dt, nt, M, eps, S, np.full(N, 10.0), U, psi0_batch=psi0, eps_bound=10.0) as p:
        p.forward(keep_for_gradient=True)
        grad = p.gradient().cpu().numpy()
        for c, j in ((0, 0), (1, 2), (2, 1), (3, 2)):
            F = []
            for s in (h, -h):
                e = eps.copy()
                e[c, j] += s
                p.set_pulses(e)
                F.append(p.forward())
            ref = -(F[0] - F[1]) / (2 * h)
            assert abs(grad[c, j] - ref) <= 1e-5 * np.abs(grad).max(), (c, j, grad[c, j], ref)
