"""Injection inside the persistent 2-D stepping for point sets that are not one
row with a point per node: many points at a node, a patch, a borehole, points all
over the grid (and so in the rows next to a band's edge), in any order.

Against the FP64 oracle, with the tolerance of the parity tests for traces
(1e-5), forward (both forms) and adjoint, on a grid that runs as bands of a
cooperative grid (397 x 401) and on one that runs as a cluster (101 x 90).

Time: a set of k points may not cost more than a few times the same call with
the points in one row.  A unit's entries are added once each, so 128 points
at a node are 128 dependent additions of a step and a patch 32 a unit: both are
well below the step itself (thousands of cycles), so a factor of 4 holds
whatever the clock; walking a unit's chain once for each of its entries took 90 and
11 times as long.
"""
import dataclasses

import numpy as np
import pytest
import torch

import oracle
from paper_2104_00794_gb300 import workloads as wl
from parity_util import host, problem, rel_l2, to_dev

pytestmark = pytest.mark.gpu


@pytest.fixture(autouse=True)
def _lib(cuda_lib):
    yield


def points(kind, nx, nz):
    rng = np.random.default_rng(7)
    if kind == "patch":
        z, x = np.meshgrid(np.arange(30, 62), np.arange(21, 53), indexing="ij")
        return rng.permutation((z * nx + x).ravel())
    if kind == "borehole":
        return np.arange(nz) * nx + nx // 3
    if kind == "doubled":
        return np.concatenate([np.arange(nz) * nx + nx // 3, np.arange(nx), np.arange(nx)])[:1024]
    if kind == "everywhere":
        return rng.permutation(nx * nz)[:1000]
    if kind == "reversed":
        return np.arange(nx)[::-1]
    if kind == "row":
        return np.arange(nx)
    return np.full(int(kind), 2 * nx + nx // 2)  # that many points at a node


KINDS = ["2", "17", "1024", "patch", "borehole", "doubled", "everywhere", "reversed"]


@pytest.mark.parametrize("kind", KINDS)
@pytest.mark.parametrize("nx,nz,order", [(397, 401, 8), (397, 401, 4), (101, 90, 8)])
def test_point_sets_against_oracle(nx, nz, order, kind):
    w = wl.small_2d(nx=nx, nz=nz, nt=42, order=order, nshots=1)
    pts = points(kind, nx, nz).astype(np.int64)[None]
    rng = np.random.default_rng(3)
    wav = np.ascontiguousarray(w.wavelet * rng.uniform(-1, 1, (1, 1, pts.shape[1])).astype(np.float32))
    w = dataclasses.replace(w, src=pts, wavelet=wav)
    ref = oracle.batch_forward(w, w.vel_true)
    for form in ("levels", "compensated"):
        p = problem(w, form=form)
        d = host(p.forward(to_dev(w.vel_true), to_dev(w.wavelet)))
        assert rel_l2(d, ref) <= 1e-5, form
        assert np.array_equal(d, host(p.forward(to_dev(w.vel_true), to_dev(w.wavelet)))), form
    # the adjoint field is read two nodes beside some of the points: further away it is below the fp32 range
    some = pts[:, [0, pts.shape[1] // 2, -1]]
    back = dataclasses.replace(w, src=some // nx * nx + (some % nx + 2) % nx, rec=pts)
    s = wl.synthetic_data(1, w.nt, pts.shape[1], seed=9)
    q = host(problem(back).adjoint(to_dev(w.vel0), to_dev(s)))
    assert rel_l2(q[0], oracle.adjoint(oracle.grid_of(back), back.src[0], back.rec[0], w.vel0, s[0])) <= 1e-5


@pytest.mark.parametrize("nx,nz", [(397, 401), (101, 90)])
def test_time_of_point_sets(nx, nz):
    def ms(kind):
        w = wl.small_2d(nx=nx, nz=nz, nt=130, order=8, nshots=1)
        w = dataclasses.replace(w, rec=points(kind, nx, nz).astype(np.int64)[None])
        p, v = problem(w), to_dev(w.vel0)
        s = to_dev(wl.synthetic_data(1, w.nt, w.rec.shape[1], seed=9))
        best = np.inf
        for _ in range(5):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            p.adjoint(v, s)
            b.record()
            torch.cuda.synchronize()
            best = min(best, a.elapsed_time(b))
        return best

    row = ms("row")
    for kind in ("128", "patch", "doubled"):
        assert ms(kind) <= 4 * row, kind
