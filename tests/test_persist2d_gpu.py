"""The persistent 2-D stepping (bands of rows in one cooperative grid, or one
cluster per shot) against the FP64 oracle, at the sizes where a split can go
wrong: last bands and chunks with a few rows, one and several passes of a CTA's
threads, order 4 and 8, the absorbing layer, more shots than fit at once, and
sources and receivers (some sharing a node) on the rows next to a band's edge.

Tolerances are those of the parity tests: 1e-5 on traces, 1e-4 on gradients.
"""
import dataclasses

import numpy as np
import pytest

import oracle
from paper_2104_00794_gb300 import api, native
from paper_2104_00794_gb300 import workloads as wl
from parity_util import host, oracle_dobs, problem, rel_l2, to_dev

pytestmark = pytest.mark.gpu


@pytest.fixture(autouse=True)
def _lib(cuda_lib):
    yield


CASES = [  # nx, nz, shots, order, sponge
    (101, 101, 1, 4, 0), (201, 45, 2, 8, 0), (397, 401, 1, 8, 0), (401, 133, 4, 4, 0), (5, 300, 2, 8, 0), (9, 3, 1, 8, 0),
    (1333, 41, 2, 8, 0), (2047, 36, 1, 4, 0), (130, 77, 20, 8, 0), (250, 97, 3, 8, 11), (66, 52, 1, 4, 9), (601, 161, 2, 8, 20),
]


def scattered(w, seed):
    """Sources and receivers on the rows around multiples of 4 and 8, some twice."""
    rng = np.random.default_rng(seed)
    rows = [r for r in (0, 3, 4, 7, 8, 9, 11, 12, 15, 16, 23, 24, 31, 32, w.nz - 1) if r < w.nz]
    def pts(n):
        z, x = rng.choice(rows, n), rng.integers(0, w.nx, n)
        p = z * w.nx + x
        p[n // 2] = p[0]
        return p
    src = np.stack([pts(5) for _ in range(w.nshots)]).astype(np.int64)
    rec = np.stack([pts(40) for _ in range(w.nshots)]).astype(np.int64)
    wav = np.ascontiguousarray(np.repeat(w.wavelet, 5, axis=2) * np.array([1.0, 0.5, -0.7, 0.3, 0.9], np.float32))
    return dataclasses.replace(w, src=src, rec=rec, wavelet=wav)


@pytest.mark.parametrize("case", CASES, ids=lambda c: "x".join(map(str, c)))
def test_against_oracle(case):
    nx, nz, shots, order, sponge = case
    w = scattered(wl.small_2d(nx=nx, nz=nz, nt=75, order=order, nshots=shots, r=4), 3)
    if sponge:
        w = wl.with_sponge(w, sponge)
    d_ref = oracle.batch_forward(w, w.vel_true)
    s = wl.synthetic_data(w.nshots, w.nt, w.rec.shape[1], seed=9)
    g = oracle.grid_of(w)
    grads = {}
    for form in ("levels", "compensated"):
        try:
            p = problem(w, form=form)
            p.workspace_bytes(native.OP_FORWARD)
        except native.TprobeError:
            assert form == "compensated"
            continue
        d = host(p.forward(to_dev(w.vel_true), to_dev(w.wavelet)))
        assert rel_l2(d, d_ref) <= 1e-5, form
        q = host(p.adjoint(to_dev(w.vel0), to_dev(s)))
        for k in range(w.nshots):
            assert rel_l2(q[k], oracle.adjoint(g, w.src[k], w.rec[k], w.vel0, s[k])) <= 1e-5, (form, k)
        spec = api.ProbeSpec(kind="rademacher", r=4, T=32, seed=w.seed)
        dobs = oracle_dobs(w)
        gp, _ = p.gradient_probed(to_dev(w.vel0), to_dev(w.wavelet), to_dev(dobs), spec)
        p.status(native.OP_GRADIENT_PROBED)
        grads[form] = host(gp)
    ref, _ = oracle.batch_gradient_probed(w, w.vel0, dobs, kind="rademacher", r=4, seed=w.seed)
    for form, gp in grads.items():
        assert rel_l2(gp, ref) <= 1e-4, form
