"""QR probes at the edges of their tiles (32 levels, 64 and 128 receivers, 4 to
32 probe columns, 1 to many parts of the time axis) against LAPACK in fp64.
Random records keep cond(Y) below 1e4, so both sides are within 1e-10 of the
exact factor, and the fp32 result is within half an ulp at 1 (6e-8) of it."""
import numpy as np
import pytest

import oracle
from paper_2104_00794_gb300 import workloads as wl
from parity_util import host, problem, to_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,nt,r,nshots", [
    (20, 31, 1, 1), (40, 33, 3, 1), (63, 64, 4, 2), (65, 100, 5, 1), (130, 161, 8, 2), (128, 97, 13, 1),
    (129, 256, 16, 3), (257, 95, 17, 1), (64, 40, 32, 1), (300, 1000, 6, 5)])
def test_qr_probes_at_tile_edges(cuda_lib, nx, nt, r, nshots):
    w = wl.small_2d(nx=nx, nz=20, nt=nt, order=8, nshots=nshots)
    d = np.random.default_rng(nx + nt).standard_normal((nshots, nt, w.nrec)).astype(np.float32)
    Q = host(problem(w).qr_probes(to_dev(d), r=r, seed=7, kind="gaussian")).astype(np.float64)
    for s in range(nshots):
        ref = oracle.qr_probes(d[s], oracle.probes("gaussian", nt, r, 7, s))
        assert np.max(np.abs(Q[s] - ref)) <= 1e-7
