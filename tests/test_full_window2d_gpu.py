"""The full-storage 2-D gradient, whose imaging terms run per window of 32
adjoint levels, against the FP64 oracle: record lengths around one and several
windows, ragged grids, both orders, the absorbing layer, sources at one node.
Tolerance: 1e-4, that of the gradients in the parity tests."""
import dataclasses

import numpy as np
import pytest

import oracle
from paper_2104_00794_gb300 import workloads as wl
from parity_util import host, problem, rel_l2, to_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,nz,nt,shots,order,sponge", [
    (67, 45, 3, 1, 8, 0), (67, 45, 4, 1, 4, 0), (130, 31, 33, 2, 8, 0), (127, 30, 34, 1, 4, 0), (60, 3, 35, 1, 8, 0),
    (257, 66, 66, 3, 8, 0), (129, 1, 67, 1, 4, 0), (90, 50, 131, 2, 8, 9)])
def test_against_oracle(cuda_lib, nx, nz, nt, shots, order, sponge):
    w = wl.small_2d(nx=nx, nz=max(nz, 4), nt=nt, order=order, nshots=shots)
    if nz < 4:  # sources and receivers on the first row
        cut = lambda v: np.ascontiguousarray(v.reshape(4, nx)[:nz])
        w = dataclasses.replace(w, nz=nz, vel_true=cut(w.vel_true), vel0=cut(w.vel0), src=w.src % nx, rec=w.rec % nx)
    if sponge:
        w = wl.with_sponge(w, sponge)
    w = dataclasses.replace(w, src=np.repeat(w.src, 2, axis=1), wavelet=np.repeat(w.wavelet, 2, axis=2))
    dobs = wl.synthetic_data(shots, nt, w.rec.shape[1], seed=4)
    g = host(problem(w).gradient_full(to_dev(w.vel0), to_dev(w.wavelet), to_dev(dobs))[0])
    assert rel_l2(g, oracle.batch_gradient_full(w, w.vel0, dobs)[0]) <= 1e-4
