"""How 2-D batches are split over the GPU (tp_sweep2d_plan): every grid that the
compensated form accepts has a plan, forward and adjoint, also the wide and
shallow ones whose levels alone fill the shared memory; those run, and agree
with the FP64 oracle (tolerances of the parity tests: 1e-5 on traces, 1e-4 on
gradients)."""
import pytest

from paper_2104_00794_gb300 import api, native
from paper_2104_00794_gb300 import workloads as wl


def grid(nx, nz, order, form, sponge=0):
    return native.tp_grid(2, nx, 1, nz, 10.0, 1e-3, 100, order, 0.0, native.TIME_FORMS[form], sponge,
                          50.0 if sponge else 0.0)


def geom(nshots, nsrc, nrec):
    return native.tp_geom(nshots, nsrc, 0x1000, nrec, 0x1000)


@pytest.mark.parametrize("order", [4, 8])
def test_every_accepted_compensated_grid_has_a_plan(order):
    """Acceptance and planning use different formulas: compared over the whole
    range of widths, at the depths around and below the last one accepted."""
    accepted = 0
    for nx in list(range(1, 64, 21)) + list(range(64, 1500, 180)) + list(range(1500, 2049, 24)) + [2047, 2048]:
        for nrec in {1, min(nx, 500), min(nx, 1024)}:
            for nshots in (1, 9):
                e = geom(nshots, 1, nrec)
                ok = lambda nz: native.tp_form_supported(grid(nx, nz, order, "compensated"), e)
                deepest = max((nz for nz in range(1, 16 * (16 if nx > 600 else 200)) if nz % 16 == 0 and ok(nz)), default=0)
                for nz in {1, 7, 33, 65, 100, deepest - 17, deepest - 1, deepest}:
                    if nz < 1 or not ok(nz):
                        continue
                    accepted += 1
                    g = grid(nx, nz, order, "compensated")
                    for adjoint in (False, True):
                        plan = native.tp_sweep2d_plan(g, e, adjoint)
                        assert plan[0] in (1, 2), (nx, nz, nrec, nshots, adjoint)
                        assert plan[1] * plan[2] >= nz and plan[4] >= 1
    assert accepted > 500


def test_plan_reports_the_per_step_path():
    assert native.tp_sweep2d_plan(grid(601, 201, 8, "increment"), geom(4, 1, 601))[0] == 0
    assert native.tp_sweep2d_plan(grid(601, 201, 8, "levels"), geom(4, 1, 1025))[0] == 0
    assert native.tp_sweep2d_plan(grid(601, 201, 8, "levels"), geom(4, 1, 601))[0] in (1, 2)
    assert native.tp_sweep2d_plan(grid(601, 201, 8, "levels", 20), geom(4, 1, 601))[0] in (1, 2)


def test_edge_words_follow_the_batch():
    """The words that bands exchange are counted for the bands a batch can have, not
    for a full GPU of the widest exchange (60 MB here, cleared by every call)."""
    small = native.tp_workspace_bytes(native.OP_FORWARD, grid(2048, 16, 8, "levels"), geom(1, 1, 1024))
    assert small <= 8 << 20
    one = native.tp_workspace_bytes(native.OP_FORWARD, grid(601, 201, 8, "levels"), geom(1, 1, 601))
    many = native.tp_workspace_bytes(native.OP_FORWARD, grid(601, 201, 8, "levels"), geom(16, 1, 601))
    assert one <= many / 4


WIDE = [  # nx, nz, shots, order, receivers: 5 to 11 rows per CTA of a cluster
    (2048, 100, 1, 8, 1024), (2048, 100, 2, 4, 1024), (2001, 101, 8, 8, 1001), (1801, 120, 1, 4, 200), (2041, 143, 1, 8, 3),
    (1855, 160, 1, 8, 5), (1689, 175, 1, 4, 7), (1613, 67, 3, 8, 900),
]


@pytest.mark.gpu
@pytest.mark.parametrize("nx,nz,nshots,order,nrec", WIDE)
def test_wide_grids_run_the_default_form(cuda_lib, nx, nz, nshots, order, nrec):
    import dataclasses

    import numpy as np

    import oracle
    from parity_util import host, oracle_dobs, problem, rel_l2, to_dev

    w = wl.small_2d(nx=nx, nz=nz, nt=41, order=order, nshots=nshots, r=4)
    rng = np.random.default_rng(nx)
    # sources and receivers on rows around the bands' edges, receivers beside a source
    rows = rng.integers(0, nz, (nshots, 3))
    src = rows * nx + rng.integers(0, nx, (nshots, 3))
    src[:, 2] = src[:, 0]  # two at a node
    rec = np.clip(src[:, rng.integers(0, 3, nrec)] + rng.integers(-9, 10, (nshots, nrec)), 0, nx * nz - 1)
    wav = np.repeat(w.wavelet, 3, axis=2) * np.array([1.0, 0.4, -0.6], np.float32)
    w = dataclasses.replace(w, src=src.astype(np.int64), rec=rec.astype(np.int64), wavelet=np.ascontiguousarray(wav))
    p = problem(w, form="auto")
    assert p.form == "compensated"
    d_ref = oracle.batch_forward(w, w.vel_true)
    assert rel_l2(host(p.forward(to_dev(w.vel_true), to_dev(w.wavelet))), d_ref) <= 1e-5
    s = wl.synthetic_data(nshots, w.nt, nrec, seed=9)
    q = host(p.adjoint(to_dev(w.vel0), to_dev(s)))
    g = oracle.grid_of(w)
    for k in range(nshots):
        assert rel_l2(q[k], oracle.adjoint(g, w.src[k], w.rec[k], w.vel0, s[k])) <= 1e-5, k
    dobs = oracle_dobs(w)
    spec = api.ProbeSpec(kind="rademacher", r=4, T=32, seed=w.seed)
    gp, _ = p.gradient_probed(to_dev(w.vel0), to_dev(w.wavelet), to_dev(dobs), spec)
    p.status(native.OP_GRADIENT_PROBED)
    ref, _ = oracle.batch_gradient_probed(w, w.vel0, dobs, kind="rademacher", r=4, seed=w.seed)
    assert rel_l2(host(gp), ref) <= 1e-4


@pytest.mark.gpu
def test_less_work_does_not_take_longer(cuda_lib):
    """A split is taken by an estimate; with a wrong one a sixth of the rows took
    as long as all of them (1500 x 60 against 1500 x 400), and one shot longer
    than sixteen (601 x 201)."""
    import dataclasses

    import torch

    from parity_util import problem, to_dev

    def ms(nx, nz, nshots):
        w = wl.small_2d(nx=nx, nz=nz, nt=200, order=8, nshots=nshots)
        w = dataclasses.replace(w, rec=w.rec[:, ::2].copy())  # at most 1024: more are stepped a launch at a time
        p, v, q = problem(w), to_dev(w.vel0), to_dev(w.wavelet)
        best = float("inf")
        for _ in range(6):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            p.forward(v, q)
            b.record()
            torch.cuda.synchronize()
            best = min(best, a.elapsed_time(b))
        return best

    assert ms(1500, 60, 1) <= 0.8 * ms(1500, 400, 1)
    assert ms(601, 201, 1) <= ms(601, 201, 16)
