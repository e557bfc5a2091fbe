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
    return [(r[0], *map(int, r[1:])) for r in rows if any(k in r[0] for k in ("fwd_kernel", "bwd_kernel", "density_kernel", "grad_"))]


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


@pytest.mark.parametrize("code", [COOPERATIVE, DENSITY], ids=["cooperative", "density_items"])
def test_routes(tmp_path, code):
    run_child(tmp_path, code)
