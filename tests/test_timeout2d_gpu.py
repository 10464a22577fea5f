"""The bounded wait of the 2-D bands for their neighbours' edge rows, made to run
out by a limit of one cycle: the call ends, reports TP_ERR_TIMEOUT and shows NaN
in every result that could be taken for a valid one, and the next call with the
default limit gives the result of a call that never timed out, bit for bit.  All
three modes (levels, compensated, absorbing layer) on grids that run as bands."""
import numpy as np
import pytest

from paper_2104_00794_gb300 import api, native
from paper_2104_00794_gb300 import workloads as wl
from parity_util import host, problem, to_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("form,sponge,call", [
    ("levels", 0, "probed"), ("compensated", 0, "probed"), ("levels", 20, "probed"), ("levels", 0, "full"),
    ("levels", 0, "forward"), ("compensated", 0, "forward"), ("levels", 0, "adjoint"), ("levels", 0, "image")])
def test_band_wait_runs_out_and_recovers(cuda_lib, form, sponge, call):
    w = wl.small_2d(nx=601 if sponge else 397, nz=201 if sponge else 401, nt=70, order=8, nshots=4)
    if sponge:
        w = wl.with_sponge(w, sponge)
    p = problem(w, form=form)
    assert native.tp_sweep2d_plan(p.grid, p.geom, call == "adjoint")[0] == 1
    vel, wav = to_dev(w.vel0), to_dev(w.wavelet)
    dobs = to_dev(wl.synthetic_data(w.nshots, w.nt, w.rec.shape[1], seed=3))
    spec = api.ProbeSpec(kind="rademacher", r=4, T=32, seed=11)
    state = p.new_state(spec)
    op = {"probed": native.OP_GRADIENT_PROBED, "full": native.OP_GRADIENT_FULL, "forward": native.OP_FORWARD,
          "adjoint": native.OP_ADJOINT, "image": native.OP_PROBED_BACKWARD}[call]

    def run():
        if call == "probed":
            return p.gradient_probed(vel, wav, dobs, spec)
        if call == "full":
            return p.gradient_full(vel, wav, dobs)
        if call == "forward":
            return (p.forward(vel, wav),)
        if call == "adjoint":
            return (p.adjoint(vel, dobs),)
        p.probed_forward(vel, wav, spec, state)
        return (p.probed_image(vel, dobs, spec, state),)

    ref = [host(t).copy() for t in run()]
    assert all(np.isfinite(r).all() for r in ref)
    p.status(op)

    native.tp_set_wait_limit(1)
    try:
        bad = [host(t).copy() for t in run()]
        with pytest.raises(native.TprobeError) as ei:
            p.status(op)
        assert ei.value.status == native.TP_ERR_TIMEOUT
    finally:
        native.tp_set_wait_limit(0)
    assert np.isnan(bad[-1]).any()  # the misfit, the samples, the image
    if call in ("probed", "full"):
        assert np.isnan(bad[1][0])

    again = [host(t) for t in run()]
    p.status(op)
    for a, r in zip(again, ref):
        assert np.array_equal(a, r)
