"""Device memory of the gradient's set-up, on the host: the library runs in a child process against a stand-in for the
CUDA runtime (host memory, kernels that do nothing) whose n-th allocation fails, or whose memory is small."""
import pytest

from fake_cudart import run_child

CHILD = r"""
import ctypes as ct, sys
import numpy as np
from paper_1801_04382_gb300 import KrotovError, Problem, cascaded_chain
fake = ct.CDLL(sys.argv[1])
N, nc, precision, strided = int(sys.argv[2]), int(sys.argv[3]), sys.argv[4], sys.argv[5] == "strided"
nt, M = 4, 2
net = cascaded_chain(N, nc)


def problem():
    eps = np.ones((N, nt))
    return Problem(net, 0.04, nt, M, eps, eps, np.full(N, 10.0), np.full((3, M, 1 + 2 * N * (nc + 1)), 0.5), precision=precision)


def gradient(p):
    out = np.zeros((N, nt))
    return p._lib.krotov_gradient(p._h, None, out.ctypes.data_as(ct.c_void_p), None)


p = problem()
n0, clean = fake.fake_mallocs(), p.info.device_bytes
p.forward(keep_for_gradient=True)
assert gradient(p) == 0
steps, full = fake.fake_mallocs() - n0, p.get_info().device_bytes
assert steps >= 7 and full > clean
p.forward(keep_for_gradient=True)
assert fake.fake_mallocs() == n0 + steps            # a second sweep allocates nothing
p.close()
for n in range(1, steps + 1):
    p = problem()
    fake.fake_fail_in(n)
    try:
        p.forward(keep_for_gradient=True)
        assert n == steps and strided, n            # no room for the series' terms: the strided kernel
        assert gradient(p) == 0
        p.close()
        continue
    except KrotovError as e:
        assert "KT_ERR_OOM" in str(e), e
    assert p.get_info().device_bytes == clean       # nothing half set up
    before, ran = fake.fake_mallocs(), fake.fake_launches()
    assert gradient(p) != 0 and fake.fake_launches() == ran
    fake.fake_fail_in(n)                            # again without room: refused again
    try:
        p.forward(keep_for_gradient=True)
        raise SystemExit(f"allocation {n}: the second call went through")
    except KrotovError as e:
        assert "KT_ERR_OOM" in str(e), e
    assert fake.fake_launches() == ran
    fake.fake_fail_in(-1)
    before = fake.fake_mallocs()
    p.forward(keep_for_gradient=True)               # with room: a set-up from the beginning
    assert fake.fake_mallocs() - before == steps and p.get_info().device_bytes == full
    assert gradient(p) == 0
    p.close()
print("ok")
"""


ROOM = r"""
import ctypes as ct, sys
import numpy as np
from paper_1801_04382_gb300 import Problem, cascaded_chain
fake = ct.CDLL(sys.argv[1])
fake.fake_set_total.argtypes = [ct.c_size_t]
fake.fake_set_total(14 << 30)
N, nc, nt, M = 3, 2, 200, 24000
eps = np.ones((N, nt))
p = Problem(cascaded_chain(N, nc), 0.025 * nt, nt, M, eps, eps, np.full(N, 10.0), np.full((1, M, 3), 0.5), precision="fp32",
            ckpt_interval=-1)
assert 0 < p.info.costate_slots <= nt               # the co-states fill what is left of the device
before = p.info.device_bytes
p.forward(keep_for_gradient=True)
terms = M * p.info.cheb_terms * 9 * 96 * 8          # the reverse kernel's: one place per element, thread and term
states = (200 // 14 + 1 + 14 + 2) * M * 729 * 8      # kept every 14 intervals, replayed, and two co-states
assert p.get_info().device_bytes - before >= states + terms, (p.get_info().device_bytes - before, states, terms)
print("ok")
"""


@pytest.mark.parametrize("N,nc,precision,fallback", [(4, 2, "fp64", "refused"), (3, 2, "fp32", "strided")])
def test_gradient_setup_is_all_or_nothing(tmp_path, N, nc, precision, fallback):
    run_child(tmp_path, CHILD, N, nc, precision, fallback)


def test_automatic_storage_leaves_room_for_the_gradient(tmp_path):
    run_child(tmp_path, ROOM)
