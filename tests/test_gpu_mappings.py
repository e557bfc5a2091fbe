"""Thread mappings and the reverse gradient at the sizes where they can go wrong, against the FP64 oracle.

Row mapping (one element per thread): one to three nodes, cutoffs 1 to 3, tiles of one and of several
trajectories with a ragged last one, several jumps per trajectory, two channels.  Block mapping (three or two
fibers per thread): four nodes in FP32-mixed.  Reverse gradient: one to four nodes, with and without jumps.
Tolerances are those of test_gpu_parity.py and test_gpu_gradient.py for the same quantities."""
import numpy as np
import pytest

import synth_inputs as si
from oracle import gradient as og
from oracle import mcwf
from oracle import model as om
from paper_1801_04382_gb300 import Problem, cascaded_chain
from test_gpu_parity import compare, run_gpu, run_oracle, setup

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,nc,M,nt,lind", [(1, 2, 33, 30, "collective"), (2, 1, 7, 40, "local"), (2, 2, 3, 24, "collective"),
                                            (2, 3, 2, 16, "local"), (3, 1, 5, 24, "collective")])
def test_row_mapping_fp64(N, nc, M, nt, lind):
    c = setup(N, nc, 0.05 * nt, nt, M, 30.0, 11 + N, 1, random_init=True, lindblad=lind)
    gpu = run_gpu(c)
    _, res = run_oracle(c)
    assert sum(len(r) for r in gpu["recs"][0]) >= 1
    compare(c, gpu, res, 1e-10, 1e-10, 1e-10, 1e-9)


@pytest.mark.parametrize("nc,M", [(1, 3), (2, 2)])
def test_block_mapping_fp32(nc, M):
    c = setup(4, nc, 0.06, 6, M, 30.0, 5, 1, random_init=True)
    gpu = run_gpu(c, "fp32")
    _, res = run_oracle(c)
    compare(c, gpu, res, 3e-5, 1e-5, 1e-4, 1e-4, margin_min=1e-5)


@pytest.mark.parametrize("N,nc,M,nt,precision,tol", [(1, 2, 3, 30, "fp64", 1e-10), (2, 2, 4, 24, "fp64", 1e-10),
                                                     (3, 1, 4, 20, "fp64", 1e-10), (4, 1, 2, 4, "fp32", 2e-4)])
def test_reverse_gradient(N, nc, M, nt, precision, tol):
    T = 0.05 * nt
    eps, S = si.guess_pulses(N, nt, T, 30.0), si.shape_functions(N, nt, T)
    U = si.uniforms(21, 2, M, 1 + 2 * N * (1 + nc))
    psi0 = si.random_states(77, M, (3 * (nc + 1)) ** N)
    with Problem(cascaded_chain(N, nc), T, nt, M, eps, S, np.full(N, 10.0), U, psi0_batch=psi0, precision=precision) as p:
        p.forward(keep_for_gradient=True)
        recs = p.records()
        grad = p.gradient().cpu().numpy()
    ref, _ = og.gradient(om.build_model(N, nc), eps, T, psi0, [[mcwf.Jump(*r) for r in rk] for rk in recs])
    assert np.abs(grad - ref).max() <= tol * np.abs(ref).max()
