"""The 2-D band kernel (bands of every shot in one cooperative grid) at grids that
the planner gives to it, which every case asserts: both orders, the absorbing
layer, last bands of a few rows, more shots than run at once, coefficients in
global memory, the imaging windows behind a band launch and a captured one; and
the path of a launch per step (more than 1024 receivers), bit for bit the same.

Against the FP64 oracle, with the tolerances of the parity tests: 1e-5 on traces,
1e-4 on gradients.
"""
import dataclasses

import numpy as np
import pytest
import torch

import oracle
from paper_2104_00794_gb300 import api, native
from paper_2104_00794_gb300 import workloads as wl
from parity_util import host, oracle_dobs, problem, rel_l2, to_dev

pytestmark = pytest.mark.gpu


@pytest.fixture(autouse=True)
def _lib(cuda_lib):
    yield


def plan(w, form="levels", adjoint=False):
    p = problem(w, form=form)
    return native.tp_sweep2d_plan(p.grid, p.geom, adjoint)


def at_band_edges(w, rpc, seed=3, nrec=60, twice=True):
    """Sources and receivers on the rows beside the bands' edges, some twice (or all different)."""
    rng = np.random.default_rng(seed)
    rows = sorted({r for k in range(0, w.nz + rpc, rpc) for r in (k - 4, k - 1, k, k + 3) if 0 <= r < w.nz} | {0, w.nz - 1})

    def pts(n):
        p = rng.choice(rows, n) * w.nx + rng.integers(0, w.nx, n)
        if twice:
            p[n // 2] = p[0]
        return p
    src = np.stack([pts(5) for _ in range(w.nshots)]).astype(np.int64)
    rec = np.stack([pts(nrec) for _ in range(w.nshots)]).astype(np.int64)
    rec[:, 1:6] = src // w.nx * w.nx + (src % w.nx + 2) % w.nx  # near every source: far ones stay below the fp32 range
    if not twice:
        rec = np.stack([np.unique(r)[:nrec - 6] for r in rec])
        src = np.stack([np.unique(s) for s in src])
    wav = np.ascontiguousarray(np.repeat(w.wavelet, 5, axis=2) * np.array([1.0, 0.5, -0.7, 0.3, 0.9], np.float32))
    return dataclasses.replace(w, src=src, rec=rec, wavelet=wav)


CASES = [  # nx, nz, shots, order, sponge, form
    (397, 401, 1, 8, 0, "levels"), (397, 401, 4, 8, 0, "compensated"), (601, 297, 2, 4, 0, "levels"),
    (601, 297, 2, 4, 0, "compensated"), (601, 201, 4, 8, 20, "levels"), (601, 201, 4, 4, 20, "levels"),
    (250, 401, 20, 8, 0, "compensated"), (397, 201, 26, 4, 12, "levels"), (1001, 393, 8, 8, 0, "levels"),
    (1001, 401, 8, 4, 0, "levels"), (801, 297, 7, 8, 0, "compensated"), (397, 386, 1, 8, 0, "levels"),
]


@pytest.mark.parametrize("case", CASES, ids=lambda c: "x".join(map(str, c)))
def test_bands_against_oracle(case):
    nx, nz, shots, order, sponge, form = case
    w = wl.small_2d(nx=nx, nz=nz, nt=45, order=order, nshots=shots, r=4)
    if sponge:
        w = wl.with_sponge(w, sponge)
    pl = plan(w, form)
    assert pl[0] == 1, pl
    w = at_band_edges(w, pl[2])
    pl = plan(w, form)
    assert pl[0] == 1 and pl[1] * pl[2] >= nz, pl
    p = problem(w, form=form)
    d = host(p.forward(to_dev(w.vel_true), to_dev(w.wavelet)))
    assert rel_l2(d, oracle.batch_forward(w, w.vel_true)) <= 1e-5
    s = wl.synthetic_data(w.nshots, w.nt, w.rec.shape[1], seed=9)
    q = host(p.adjoint(to_dev(w.vel0), to_dev(s)))
    g = oracle.grid_of(w)
    for k in range(shots):
        assert rel_l2(q[k], oracle.adjoint(g, w.src[k], w.rec[k], w.vel0, s[k])) <= 1e-5, k


def test_cases_cover_the_kinds_of_bands():
    """Rounds of shots, last bands of a few rows, both march lengths, c2 in global memory."""
    plans = []
    for nx, nz, shots, order, sponge, form in CASES:
        w = wl.small_2d(nx=nx, nz=nz, nt=45, order=order, nshots=shots, r=4)
        pl = plan(wl.with_sponge(w, sponge) if sponge else w, form)
        plans.append((nz - (pl[1] - 1) * pl[2], shots > pl[4], *pl))
    assert any(last <= 2 for last, *_ in plans)
    assert any(rounds for _, rounds, *_ in plans)
    assert {pl[5] for pl in plans} == {4, 8}
    assert {pl[7] for pl in plans} == {0, 1}


@pytest.mark.parametrize("nx,nz,shots,order,sponge", [(397, 401, 2, 8, 0), (601, 201, 4, 8, 20), (601, 297, 1, 4, 0)])
def test_gradients_behind_band_launches(nx, nz, shots, order, sponge):
    """Full storage (imaging windows of 32 levels, with a ragged tail) and probed."""
    w = wl.small_2d(nx=nx, nz=nz, nt=75, order=order, nshots=shots, r=4)
    if sponge:
        w = wl.with_sponge(w, sponge)
    assert plan(w)[0] == 1 and plan(w, adjoint=True)[0] == 1
    w = at_band_edges(w, plan(w)[2])
    dobs = oracle_dobs(w)
    p = problem(w)
    args = (to_dev(w.vel0), to_dev(w.wavelet), to_dev(dobs))
    g = host(p.gradient_full(*args)[0])
    assert rel_l2(g, oracle.batch_gradient_full(w, w.vel0, dobs)[0]) <= 1e-4
    spec = api.ProbeSpec(kind="rademacher", r=4, T=32, seed=w.seed)
    g = host(p.gradient_probed(*args, spec)[0])
    ref, _ = oracle.batch_gradient_probed(w, w.vel0, dobs, kind="rademacher", r=4, seed=w.seed)
    assert rel_l2(g, ref) <= 1e-4


def test_captured_band_launches():
    """A captured gradient on a band grid: replays equal the eager call bit for bit, on two streams too."""
    w = wl.small_2d(nx=397, nz=401, nt=75, order=8, nshots=4, r=4)
    assert plan(w, "compensated")[0] == 1 and plan(w, adjoint=True)[0] == 1
    p = problem(w, form="compensated")
    spec = api.ProbeSpec(kind="rademacher", r=4, T=32, seed=3)
    args = (to_dev(w.vel0), to_dev(w.wavelet), to_dev(wl.synthetic_data(4, w.nt, w.rec.shape[1], seed=2)))
    ref = [host(t).copy() for t in p.gradient_probed(*args, spec)]
    graphs = [api.GraphedGradient(problem(w, form="compensated"), spec) for _ in range(2)]
    streams = [torch.cuda.Stream() for _ in range(2)]
    for _ in range(3):
        for gr, st in zip(graphs, streams):
            with torch.cuda.stream(st):
                gr(*args)
    for gr in graphs:
        torch.cuda.synchronize()
        assert np.array_equal(host(gr.grad), ref[0])


def many_receivers(w):
    """The same receivers and copies of them, more than one launch's lists hold."""
    times = 1100 // w.rec.shape[1] + 1
    return dataclasses.replace(w, rec=np.tile(w.rec, (1, times)))


STEPS = [(150, 90, 2, 8, 0), (150, 90, 2, 4, 0), (150, 90, 1, 8, 12), (397, 401, 1, 8, 20), (397, 401, 1, 4, 0)]


@pytest.mark.parametrize("nx,nz,shots,order,sponge", STEPS)
def test_launch_per_step_equals_the_persistent_path(nx, nz, shots, order, sponge):
    """Traces of the two paths, with and without the layer, bit for bit (the
    layer's quotient against a division: the field runs down to subnormal values
    ahead of the wave).  All points differ: entries that share a node are added
    with other roundings by a launch per step."""
    w = wl.small_2d(nx=nx, nz=nz, nt=300, order=order, nshots=shots)
    if sponge:
        w = wl.with_sponge(w, sponge)
    w = at_band_edges(w, 8, twice=False)
    n = w.rec.shape[1]
    assert plan(w)[0] in (1, 2) and plan(many_receivers(w))[0] == 0
    a = host(problem(w).forward(to_dev(w.vel_true), to_dev(w.wavelet)))
    b = host(problem(many_receivers(w)).forward(to_dev(w.vel_true), to_dev(w.wavelet)))
    for i in range(0, b.shape[2], n):
        assert np.array_equal(a, b[:, :, i:i + n])
    s = wl.synthetic_data(shots, w.nt, n, seed=9)
    more = np.stack([np.concatenate([r, np.setdiff1d(np.arange(w.nx * w.nz), r)[:1100]]) for r in w.rec])
    sz = np.zeros((shots, w.nt, more.shape[1]), np.float32)
    sz[:, :, :n] = s  # the others radiate nothing
    assert np.array_equal(host(problem(w).adjoint(to_dev(w.vel0), to_dev(s))),
                          host(problem(dataclasses.replace(w, rec=more)).adjoint(to_dev(w.vel0), to_dev(sz))))


@pytest.mark.parametrize("sponge", [0, 9])
def test_launch_per_step_against_oracle(sponge):
    """More than 1024 receivers, every node of them shared: adjoint, full and
    probed gradient in the levels form, the forward repeated bit for bit."""
    w = wl.small_2d(nx=90, nz=50, nt=75, order=8, nshots=2, r=4)
    if sponge:
        w = wl.with_sponge(w, sponge)
    w = many_receivers(at_band_edges(w, 8))
    assert plan(w)[0] == 0
    p = problem(w)
    d = host(p.forward(to_dev(w.vel_true), to_dev(w.wavelet)))
    assert np.array_equal(d, host(p.forward(to_dev(w.vel_true), to_dev(w.wavelet))))
    assert rel_l2(d, oracle.batch_forward(w, w.vel_true)) <= 1e-5
    s = wl.synthetic_data(2, w.nt, w.rec.shape[1], seed=9)
    q = host(p.adjoint(to_dev(w.vel0), to_dev(s)))
    for k in range(2):
        assert rel_l2(q[k], oracle.adjoint(oracle.grid_of(w), w.src[k], w.rec[k], w.vel0, s[k])) <= 1e-5
    dobs = oracle_dobs(w)
    args = (to_dev(w.vel0), to_dev(w.wavelet), to_dev(dobs))
    assert rel_l2(host(p.gradient_full(*args)[0]), oracle.batch_gradient_full(w, w.vel0, dobs)[0]) <= 1e-4
    spec = api.ProbeSpec(kind="rademacher", r=4, T=32, seed=w.seed)
    ref, _ = oracle.batch_gradient_probed(w, w.vel0, dobs, kind="rademacher", r=4, seed=w.seed)
    assert rel_l2(host(p.gradient_probed(*args, spec)[0]), ref) <= 1e-4


KINDS = [  # nx, nz, shots, order, sponge, form -> bands (1) or clusters (2), rows per march, c2 in shared memory
    (1300, 17, 1, 4, 0, "compensated", 2, 2, 1), (1500, 41, 1, 4, 0, "compensated", 2, 4, 0),
    (1500, 100, 1, 4, 0, "compensated", 1, 4, 0), (601, 17, 1, 8, 0, "compensated", 2, 2, 1),
    (1800, 77, 1, 8, 0, "compensated", 2, 4, 0), (1300, 41, 1, 8, 0, "compensated", 2, 4, 1),
    (1500, 150, 1, 8, 0, "compensated", 1, 4, 0), (1300, 17, 1, 4, 0, "levels", 2, 2, 1),
    (2045, 100, 1, 4, 0, "levels", 2, 4, 0), (1500, 41, 3, 4, 0, "levels", 2, 4, 1), (2045, 150, 1, 4, 0, "levels", 1, 4, 0),
    (1001, 17, 9, 8, 0, "levels", 2, 2, 1), (1500, 41, 1, 8, 0, "levels", 2, 4, 0), (1300, 41, 1, 8, 0, "levels", 2, 4, 1),
    (2045, 150, 1, 8, 0, "levels", 1, 4, 0), (2045, 100, 1, 8, 10, "levels", 1, 4, 0), (2045, 100, 1, 4, 10, "levels", 1, 4, 0),
    (1001, 17, 1, 8, 10, "levels", 2, 2, 1), (601, 100, 1, 8, 10, "levels", 2, 4, 1), (1300, 17, 1, 4, 10, "levels", 2, 2, 1),
]


@pytest.mark.parametrize("kind", KINDS, ids=lambda c: "x".join(map(str, c)))
def test_every_kind_of_split_against_oracle(kind):
    """Wide grids, where the planner takes the marches and the places of c2 that the
    other tests do not: clusters of two and four rows a march, lean ones, bands
    with c2 in global memory; points beside the CTAs' edges, in a patch, in a row."""
    nx, nz, shots, order, sponge, form, *want = kind
    w = wl.small_2d(nx=nx, nz=nz, nt=41, order=order, nshots=shots)
    if sponge:
        w = wl.with_sponge(w, sponge)
    w = at_band_edges(w, 4)
    pl = plan(w, form)
    assert [pl[0], pl[3], pl[5]] == want, pl
    patch = ((np.arange(5, 13)[:, None] % nz) * nx + nx // 2 + np.arange(9)).ravel()
    row = 3 * nx + np.arange(nx // 2 - 40, nx // 2 + 40)
    w = dataclasses.replace(w, rec=np.concatenate([w.rec, np.tile(np.concatenate([patch, row]), (shots, 1))], axis=1))
    p = problem(w, form=form)
    d = host(p.forward(to_dev(w.vel_true), to_dev(w.wavelet)))
    assert rel_l2(d, oracle.batch_forward(w, w.vel_true)) <= 1e-5
    s = wl.synthetic_data(shots, w.nt, w.rec.shape[1], seed=9)
    q = host(p.adjoint(to_dev(w.vel0), to_dev(s)))
    for k in range(shots):
        assert rel_l2(q[k], oracle.adjoint(oracle.grid_of(w), w.src[k], w.rec[k], w.vel0, s[k])) <= 1e-5, k
    back = dataclasses.replace(w, src=w.rec, rec=w.src,
                               wavelet=np.ascontiguousarray(np.repeat(w.wavelet[:, :, :1], w.rec.shape[1], axis=2)))
    if form == "compensated":  # the points inject in the compensated form too
        d = host(problem(back, form=form).forward(to_dev(w.vel_true), to_dev(back.wavelet)))
        assert rel_l2(d, oracle.batch_forward(back, w.vel_true)) <= 1e-5
