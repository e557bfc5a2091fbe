"""Which kernels a problem launches, on the host against a stand-in for the CUDA runtime (fake_cudart.py)."""
import pytest

from fake_cudart import run_child

HEAD = r"""
import ctypes as ct, sys
import numpy as np
from paper_1801_04382_gb300 import Batch, DensityProblem, Problem, _capi, cascaded_chain
from paper_1801_04382_gb300.problem import _descriptors
fake = ct.CDLL(sys.argv[1])
fake.fake_log.restype = ct.c_char_p


def launched(fn):
    '''[(kernel, grid, block, shared bytes, cooperative, cluster size)] of the sweep kernels that fn launches'''
    fake.fake_log_clear()
    fn()
    rows = [ln.split() for ln in fake.fake_log().decode().splitlines()]
    return [(r[0], *map(int, r[1:])) for r in rows if any(k in r[0] for k in ("fwd_kernel", "bwd_kernel", "density_kernel", "grad_kernel", "grad_adj_kernel"))]


def spec(n, nc, nt, M, **more):
    eps = np.ones((n, nt))
    return dict(dict(net=cascaded_chain(n, nc), T=0.05 * nt, nt=nt, M=M, eps_guess=eps, shape=eps, lam=np.full(n, 10.0),
                     uniforms=np.full((3, M, 1 + 2 * n * (nc + 1)), 0.5)), **more)
"""

COOPERATIVE = HEAD + r"""
p = Problem(**spec(2, 2, 4, 3))
assert p.info.whole_sweep == 1
guess, back = launched(lambda: p.forward()), launched(lambda: p.backward())
update = launched(lambda: p.forward(update=True))
assert len(guess) == len(back) == len(update) == 1
# the updating sweep's CTAs wait for one another: all of them resident; nothing waits in the others
assert (guess[0][4], back[0][4], update[0][4]) == (0, 0, 1), (guess, back, update)
b = Batch([spec(2, 2, 4, 3), spec(2, 1, 6, 2), spec(3, 1, 4, 2)])
rows = launched(lambda: b.update(1))
assert rows and all(r[4] == 0 for r in rows), rows
print("ok")
"""

DENSITY = HEAD + r"""
def density(items):
    s = spec(2, 1, 4, 1, uniforms=np.full((1, 1, 1), -1.0))
    keep, md, cfg = _descriptors(s["net"], s["T"], s["nt"], 1, s["eps_guess"], s["shape"], s["lam"], s["uniforms"],
                                 items_per_thread=items)
    lib, h = _capi.load(), ct.c_void_p()
    assert lib.krotov_init_density(ct.byref(md), ct.byref(cfg), None, ct.byref(h)) == 0
    info = _capi.Info()
    assert lib.krotov_get_info(h, ct.byref(info)) == 0
    rows = launched(lambda: lib.propagate_forward(h, 0, None, None))
    lib.krotov_free(h)
    return info, rows


info, rows = density(0)
assert rows and all("density_kernel" in r[0] and r[5] == 4 for r in rows), rows
for items in (4, 8):
    info, rows = density(items)
    assert info.items_per_thread == items
    assert rows and all("fwd_kernelIdLi%dELi0" % items in r[0] for r in rows), rows
print("ok")
"""


KERNELS = HEAD + r"""
import cmath


def kernel(net, nt, M, how="forward", **more):
    s = spec(net.n_nodes, 1, nt, M, net=net, **more)
    with Problem(**s) as p:
        if how == "forward":
            rows = launched(lambda: p.forward())
        elif how == "kept":
            rows = launched(lambda: p.forward(keep_for_gradient=True))
        else:
            p.forward(keep_for_gradient=True)
            out = np.zeros((net.n_nodes, nt))
            rows = launched(lambda: p._lib.krotov_gradient(p._h, None, out.ctypes.data_as(ct.c_void_p), None))
    assert rows, how
    names = {r[0].split("EEEv")[0].replace("_ZN2kt", "").lstrip("0123456789") for r in rows}
    assert len(names) == 1 or how == "gradient", names
    return names if how == "gradient" else names.pop()


def plain(N, nc):
    net = cascaded_chain(N, nc)
    x = np.zeros((net.n_loc, net.n_loc), dtype=complex)
    x[0, nc + 1] = x[nc + 1, 0] = 0.4
    net.h0_local = net.h0_local + x
    return net


def phase(N, nc):
    return cascaded_chain(N, nc, g=cmath.exp(0.2j * cmath.pi))


T = {"fp32": "f", "fp64": "d"}
for prec in ("fp32", "fp64"):
    t = T[prec]
    # fibers: plain, complex cavity structure (tile width 1 compiled in for n_loc = 9), real / imaginary
    assert kernel(plain(2, 1), 4, 5, tile_traj=2, precision=prec).startswith(f"fwd_kernelI{t}Li6ELi6ELi0ELb0")
    assert kernel(plain(2, 2), 4, 5, tile_traj=1, precision=prec).startswith(f"fwd_kernelI{t}Li9ELi9ELi0ELb0")
    assert kernel(phase(2, 1), 4, 5, tile_traj=1, precision=prec).startswith(f"fwd_kernelI{t}Li6ELi6ELi1ELb0")
    assert kernel(phase(2, 2), 4, 5, tile_traj=2, precision=prec).startswith(f"fwd_kernelI{t}Li9ELi9ELi1ELb0")
    assert kernel(phase(2, 2), 4, 5, tile_traj=1, precision=prec).startswith(f"fwd_kernelI{t}Li9ELi9ELi2ELb0")
    assert kernel(cascaded_chain(3, 1), 4, 5, tile_traj=2, precision=prec).startswith(f"fwd_kernelI{t}Li6ELi6ELi3ELb0")
    # gradient: strided where the couplings are complex, reverse where they are not
    assert any(k.startswith(f"grad_kernelI{t}Li4") for k in kernel(phase(2, 1), 4, 3, "gradient", precision=prec))
    assert all(k.startswith(f"grad_adj_kernelI{t}Li2") for k in kernel(cascaded_chain(3, 2), 4, 3, "gradient", precision=prec))
# tile loops: two CTAs of 448 threads per SM where the kernel's 72 registers leave room for them
with Problem(**spec(4, 1, 3, 1024, precision="fp32")) as p:
    p.forward()
    assert all(r[1:3] == (304, 448) for r in launched(lambda: p.backward()))
# FP32 fibers and blocks: the T form; sweeps that keep states for the gradient: the y form (codes 8 higher)
assert kernel(cascaded_chain(3, 2), 4, 5, precision="fp32").startswith("fwd_kernelIfLi9ELi9ELi4ELb0")
assert kernel(cascaded_chain(3, 2), 4, 5, "kept", precision="fp32").startswith("fwd_kernelIfLi9ELi9ELi12ELb0")
assert kernel(cascaded_chain(4, 1), 4, 5, precision="fp32").startswith("fwd_kernelIfLi12ELi6ELi5ELb0")
assert kernel(cascaded_chain(4, 1), 4, 5, "kept", precision="fp32").startswith("fwd_kernelIfLi12ELi6ELi13ELb0")
assert kernel(cascaded_chain(3, 2), 4, 5, precision="fp64").startswith("fwd_kernelIdLi1ELi0ELi7ELb0")
assert all(k.startswith("grad_adj_kernelIdLi2ELi736") for k in kernel(cascaded_chain(4, 2), 3, 2, "gradient", precision="fp64"))
print("ok")
"""


@pytest.mark.parametrize("code", [COOPERATIVE, DENSITY, KERNELS], ids=["cooperative", "density_items", "kernels"])
def test_routes(tmp_path, code):
    run_child(tmp_path, code)
