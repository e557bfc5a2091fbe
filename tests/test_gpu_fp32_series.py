"""FP32 fibers and blocks: the propagated state is that of the T form of the series in float32 arithmetic.

The norm of a state decides in which interval its trajectory jumps, so its rounding has to stay what it is.  The
reference runs the series in numpy, each FMA as a float64 product and sum rounded to float32.  Rounding twice differs
from rounding once in one case out of 2^29 or so, less than one element of one term here, by an ulp of that element;
four ulps of a unit norm are allowed."""
import numpy as np
import pytest

from paper_1801_04382_gb300 import Problem, bessel_j, cascaded_chain

pytestmark = pytest.mark.gpu

TOL = 4 * 2.0 ** -24
F = np.float32


def fma(a, b, c):
    return (a.astype(np.float64) * b.astype(np.float64) + c.astype(np.float64)).astype(F)


def cmul(ax, ay, bx, by):
    return fma(ax, bx, -(ay * by)), fma(ay, bx, ax * by)


class Series:
    """2 (G - c) / r of a cascaded chain as (offset, coefficient, imaginary?) per row and slot, in the order in which
    the kernels add a row's terms."""

    def __init__(self, net, c, r):
        self.n, self.nl, self.d = net.n_nodes, net.n_loc, net.d
        n, nl = self.n, self.nl
        self.c, self.r, self.net, x = c, r, net, np.arange(self.d)
        self.stride = [nl ** (n - 1 - i) for i in range(n)]
        self.dig = [(x // s) % nl for s in self.stride]
        a = net.a_local
        loc = [net.h0_local[i] + sum(-0.5j * abs(l[i]) ** 2 for l in net.lind_coef) * (a.conj().T @ a) for i in range(n)]
        coef = {}
        for q in range(len(net.pair_dst)):
            k = (int(net.pair_dst[q]), int(net.pair_src[q]))
            coef[k] = coef.get(k, 0.0) + net.pair_coef[q]
        for l in net.lind_coef:
            for i in range(n):
                for j in range(n):
                    if i != j and l[i] * l[j] != 0.0:
                        coef[i, j] = coef.get((i, j), 0.0) - 0.5j * np.conj(l[i]) * l[j]
        self.loc, self.pairs = loc, [(k, v) for k, v in coef.items() if abs(v) > 1e-13]
        dx, dy = np.zeros(self.d, F), np.zeros(self.d, F)
        for i in range(n):
            v = (np.diag(loc[i]) - (c if i == 0 else 0.0)) * (2.0 / r)
            dx, dy = dx + v.real.astype(F)[self.dig[i]], dy + v.imag.astype(F)[self.dig[i]]
        self.dx, self.dy = dx, dy
        self.hops = []
        up, s2 = np.diag(a, 1), np.append(np.diag(a, 1), 0.0).real       # a[x, x + 1]
        assert np.count_nonzero(a) == np.count_nonzero(up)
        ladder = {"lower": s2, "raise": np.append(0.0, up).real}         # row x <- column x + 1, x - 1
        for (i, j), v in self.pairs:
            vi, vj = ladder["raise"][self.dig[i]], ladder["lower"][self.dig[j]]
            k, last = (v * 2.0 / r).imag, n - 1
            if i == last:
                w = (F(k) * vj.astype(F)) * vi.astype(F)
            elif j == last:
                w = (F(k) * vi.astype(F)) * vj.astype(F)
            else:
                w = (k * vi * vj).astype(F)
            on = w != 0
            self.hops.append((np.where(on, x - self.stride[i] + self.stride[j], x), np.where(on, w, F(0)), True))

    def slots(self, eps):
        out, x, n, nl = [], np.arange(self.d), self.n, self.nl
        for i in [n - 1] + list(range(n - 1)):
            h = self.loc[i].astype(complex)
            for c, node in enumerate(self.net.ctrl_node):
                if node == i:
                    h = h + eps[c] * self.net.hc_local[c]
            h = h * (2.0 / self.r)
            h = h - np.diag(np.diag(h))
            for imag, part in ((False, h.real), (True, h.imag)):
                assert (np.count_nonzero(part, axis=1) <= 1).all()
                col = np.where(part.any(axis=1), np.abs(part).argmax(axis=1), np.arange(nl))
                w = part[np.arange(nl), col] * (col != np.arange(nl))
                g = self.dig[i]
                out.append((x + (col[g] - g) * self.stride[i], w.astype(F)[g], imag))
        return out + self.hops

    def twice_g(self, slots, vx, vy):
        ox, oy = cmul(self.dx, self.dy, vx, vy)
        for col, w, imag in slots:
            if imag:
                ox, oy = fma(-w, vy[col], ox), fma(w, vx[col], oy)
            else:
                ox, oy = fma(w, vx[col], ox), fma(w, vy[col], oy)
        return ox, oy

    def step(self, eps, coef, vx, vy):
        s = self.slots(eps)
        ax, ay = cmul(coef[0][0], coef[0][1], vx, vy)
        px, py, qx, qy = None, None, vx, vy
        for k in range(1, len(coef)):
            tx, ty = self.twice_g(s, qx, qy)
            tx, ty = (F(0.5) * tx, F(0.5) * ty) if k == 1 else (tx - px, ty - py)
            px, py, qx, qy = qx, qy, tx, ty
            cx, cy = coef[k]
            ax, ay = fma(-cy, ty, fma(cx, tx, ax)), fma(cy, tx, fma(cx, ty, ay))
        return ax, ay


def emulate(net, info, dt, eps, psi):
    c, r = 0.5 * (info.e_min + info.e_max), 0.5 * (info.e_max - info.e_min) * 1.0001 + 1e-12
    J = bessel_j(r * dt, 256)[:info.cheb_terms]
    ph = np.exp(-1j * c * dt)
    coef = []
    for k, j in enumerate(J):
        v = (1.0 if k == 0 else 2.0) * j * [1, -1j, -1, 1j][k % 4] * ph
        coef.append((np.full(1, v.real, F), np.full(1, v.imag, F)))
    g = Series(net, c, r)
    x, y = psi.real.astype(F), psi.imag.astype(F)
    for q in range(eps.shape[1]):
        x, y = g.step(eps[:, q], coef, x, y)
    return x.astype(np.float64) + 1j * y


@pytest.mark.parametrize("n,nc,nt,dt,tile", [(3, 2, 60, 0.025, 0), (3, 2, 20, 0.025, 4), (4, 1, 40, 0.01, 0), (4, 2, 40, 0.01, 0)])
def test_state_is_the_float32_series(n, nc, nt, dt, tile):
    net = cascaded_chain(n, nc)
    nl = net.n_loc
    psi = np.zeros(net.d, dtype=np.complex128)
    e = (nc + 1) * nl ** (n - 1)
    psi[[e, 2 * e, e + nl ** (n - 2)]] = np.sqrt([0.63, 0.07, 0.3])   # an e-r coherence and a photon in flight
    net.psi0 = psi
    t = (np.arange(nt) + 0.5) / nt
    eps = np.stack([np.sin(np.pi * t) ** 2 * (1.0 + 0.1 * i) + 0.05 * i for i in range(n)])
    U = np.full((1, 2, 1 + 2 * n * (nc + 1)), 1e-9)                   # no jump
    with Problem(net, nt * dt, nt, 2, eps, np.ones_like(eps), np.full(n, 10.0), U, precision="fp32", tile_traj=tile) as p:
        p.forward()
        z = p.states()
        ref = emulate(net, p.info, dt, eps, psi)
    assert (z[0] == z[1]).all()
    assert np.abs(z[0] - ref).max() <= TOL
    assert abs((np.abs(z[0]) ** 2).sum() - (np.abs(ref) ** 2).sum()) <= TOL
